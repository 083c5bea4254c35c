"""Timed workloads of the framework, each one pass through its public entry
points (``paper_1709_10187_gb300.rddmc`` and ``.learned``).

Kinds of case:

* ``run``       walk packets from the source to escape (``Problem.run``);
* ``slices``    a checkpointed walk: one launch from the source that advances
                every packet by ``steps`` transitions and saves it, one that
                resumes it, then the tallies and a sample of the saved states;
* ``time``      the time-dependent walk, one launch per step (``time_run``);
* ``batch``     many independent media in one graph replay (``Batch``);
* ``network``   the exit-proposal network: a training step (loss, gradients,
                Adam) or the logits of a batch;
* ``passages``  first passages of packets through regions of a medium, the
                training data of that network;
* ``setup``     from the description of a medium to the first tallies of a
                frequency-grouped hybrid walk: grid, leakage table,
                redistribution thresholds, short walk.

``transitions`` is the number of packet transitions one pass makes, known from
the slices or estimated from 1.7 tau0 / dx^2 transitions per escaping packet
(a packet scatters about 1.6 tau0 times before it leaves a slab, and each
scattering's unit frequency step is 1 / dx^2 hops between bins dx wide).
"""
import math

import numpy as np
import torch

from paper_1709_10187_gb300 import learned as L
from paper_1709_10187_gb300 import rddmc as R
from paper_1709_10187_gb300 import workloads as W

SAMPLE = 4096          # saved packet states read back by a checkpointed walk
OPS = 25               # integer operations a transition cannot do without (a quarter Philox call, the choice, the move)


def _case(kind, **kw):
    base = dict(kind=kind, ndim=1, cells=64, bins=128, xmax=30.0, tau0=1.0e5, T=1.0e4, vmax=0.0, core=0.0,
                clumpy=False, hybrid=False, dust=0.0, weights=False, packets=0, steps=0, transitions=0.0)
    base.update(kw)
    return base


def listed():
    c1, c2, wc, c3, p2 = W.C1, W.C2, W.C2_WIDECORE, W.C3_V20, W.P2
    return [
        # a small exploratory slab walked to the end: the latency of one call
        _case("run", name="slab_8x16_run", cells=8, bins=16, xmax=8.0, tau0=200.0, packets=2048,
              transitions=2048 * 590.0),
        # the tau0 = 1e5 slab of the parity configuration, every packet to escape:
        # the slowest packets set the time
        _case("run", name="slab_64x128_run", cells=c1.n[0], bins=c1.J, xmax=c1.x_max, tau0=c1.tau0,
              packets=c1.packets, transitions=c1.packets * 8.7e5),
        # the headline slab (tau0 = 1e7), a long job in checkpointed slices
        _case("slices", name="slab_256x512_slices", cells=c2.n[0], bins=c2.J, xmax=c2.x_max, tau0=c2.tau0,
              packets=4_000_000, steps=4096, transitions=4_000_000 * 8192.0),
        # the same slab on the recommended wide-core frequency grid, to escape
        _case("run", name="slab_widecore_run", cells=wc.n[0], bins=wc.J, xmax=wc.x_max, tau0=wc.tau0,
              core=wc.core_half, packets=2_000_000, transitions=2_000_000 * 2.1e4),
        # a sphere in Hubble-like outflow (20 km/s), checkpointed
        _case("slices", name="sphere_outflow_slices", ndim=3, cells=c3.n[0], bins=c3.J, xmax=c3.x_max, tau0=c3.tau0,
              vmax=c3.vmax_kms, packets=1_000_000, steps=4096, transitions=1_000_000 * 8192.0),
        # a turbulent lognormal medium, every cell its own rows (a table larger
        # than L2), long slices that carry the packets through many cells
        _case("slices", name="clumpy_cells_slices", ndim=3, cells=32, bins=128, xmax=128.0, tau0=1.0e7, clumpy=True,
              packets=100_000, steps=65536, transitions=100_000 * 131072.0),
        # continuous MC in the thin wings of the headline slab (hybrid scheme)
        _case("slices", name="slab_hybrid_slices", cells=c2.n[0], bins=c2.J, xmax=c2.x_max, tau0=c2.tau0,
              hybrid=True, packets=500_000, steps=4096, transitions=500_000 * 8192.0),
        # the paper's time-dependent resonant test (1e7 packets), its first 20 steps
        _case("time", name="time_resonant", cells=p2.n[0], bins=p2.J, xmax=p2.x_max, tau0=p2.tau0, T=p2.T,
              packets=10_000_000, steps=20, dt=1.0, leaks=False, transitions=10_000_000 * 20 * 5.7),
        # a parameter study: 64 slabs and spheres of different depth, temperature
        # and size, watchdog at 32768 transitions, replayed as one graph
        _case("batch", name="batch_64_graph", instances=64, scale=0.02, steps=32768, transitions=64 * 4000 * 26000.0),
        # one optimiser step of the proposal network at its training batch
        _case("network", name="network_train_step", train=True, bins=256, side=6, rows=8192),
        # training data of the proposal: first passages out of 6^3 regions of a
        # turbulent medium
        _case("passages", name="region_passages", ndim=3, cells=32, bins=64, xmax=64.0, tau0=1.0e6, clumpy=True,
              brick=8, margin=1, packets=200_000, transitions=200_000 * 1.0e4),
        # a new moving medium with thin wings, from its description to tallies
        _case("setup", name="medium_setup", ndim=3, cells=16, bins=64, xmax=32.0, tau0=1.0e5, clumpy=True,
              hybrid=True, packets=4096, steps=256, transitions=4096 * 256.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _slab_or_sphere(rng):
    """Geometry and medium of a drawn walk: slabs and spheres, thin to thick."""
    if rng.random() < 0.6:
        cells, bins, ndim = int(round(_log(rng, 8, 256))), int(round(_log(rng, 16, 512))), 1
    else:
        cells, bins, ndim = int(round(_log(rng, 8, 64))), int(round(_log(rng, 16, 256))), 3
    vmax = round(_log(rng, 5.0, 200.0), 2) if ndim == 3 and rng.random() < 0.5 else 0.0
    # at least 6 Doppler widths, so that the grid ends in the wings
    return dict(ndim=ndim, cells=cells, bins=bins, xmax=round(max(6.0, bins * rng.uniform(0.12, 0.6)), 2), vmax=vmax)


def draw(rng):
    kind = rng.choice(["run", "run", "slices", "slices", "time", "batch", "network", "passages", "setup"])
    if kind == "run":
        g = _slab_or_sphere(rng)
        dx = 2.0 * g["xmax"] / g["bins"]
        tau0 = round(_log(rng, 200.0, min(1.0e5, 4.0e5 * dx * dx)), 1)
        per = 1.7 * tau0 / (dx * dx) + g["cells"] ** 2
        n = int(min(_log(rng, 1000, 100_000), 5.0e10 / per))
        dust = round(rng.uniform(0.1, 5.0), 2) if rng.random() < 0.3 else 0.0
        return _case("run", tau0=tau0, packets=n, dust=dust, weights=bool(dust > 0.0 and rng.random() < 0.5),
                     transitions=n * per, **g)
    if kind == "slices":
        g = _slab_or_sphere(rng)
        steps = 4 * int(_log(rng, 64, 2048))
        n = int(_log(rng, 10_000, 1_000_000))
        return _case("slices", tau0=round(_log(rng, 1.0e4, 1.0e8), 1), packets=n, steps=steps,
                     hybrid=rng.random() < 0.25 and g["ndim"] == 1, transitions=2.0 * n * steps, **g)
    if kind == "time":
        grey = rng.random() < 0.3
        cells, bins = int(_log(rng, 31, 201)), 1 if grey else int(_log(rng, 9, 101))
        n, steps = int(_log(rng, 10_000, 4_000_000)), rng.randint(2, 16)
        return _case("time", cells=cells, bins=bins, xmax=5.0 if grey else 2500.0, T=1.0e4 if grey else 10.0,
                     tau0=1.0e3 if grey else W.P2.tau0, packets=n, steps=steps,
                     dt=round(rng.uniform(0.02, 0.2) if grey else rng.uniform(0.5, 2.0), 3),
                     leaks=rng.random() < 0.3, transitions=n * steps * 6.0)
    if kind == "batch":
        inst, steps = rng.randint(2, 96), 4 * int(_log(rng, 256, 8192))
        scale = round(_log(rng, 0.002, 0.02), 4)
        return _case("batch", instances=inst, scale=scale, steps=steps, transitions=inst * 2.0e5 * scale * steps * 0.8)
    if kind == "network":
        return _case("network", train=rng.random() < 0.5, bins=rng.choice([16, 37, 64, 128, 256]),
                     side=rng.choice([2, 4, 6, 14]), rows=64 * int(_log(rng, 1, 256)))
    if kind == "passages":
        n = int(_log(rng, 2000, 200_000))
        return _case("passages", ndim=3, cells=rng.choice([16, 24, 32]), bins=64, xmax=64.0,
                     tau0=round(_log(rng, 1.0e5, 1.0e6), 1), clumpy=True, brick=8, margin=rng.choice([1, 2]), packets=n,
                     transitions=n * 1.0e4)
    return _case("setup", ndim=3, cells=rng.randint(8, 16), bins=rng.randint(16, 64),
                 xmax=round(rng.uniform(16.0, 40.0), 2), tau0=round(_log(rng, 3.0e3, 1.0e5), 1), clumpy=True, hybrid=True,
                 packets=int(_log(rng, 256, 4096)), steps=256, transitions=4096 * 256.0)


# ----------------------------------------------------------------------------- inputs
def _philox_seed(seed):
    return (0x5EED << 32) + 2 * int(seed) + 1


def _workload(c):
    n = (c["cells"],) * 3 if c["ndim"] == 3 else (c["cells"], 1, 1)
    return W.Workload("case", c["ndim"], n, c["bins"], -c["xmax"], c["xmax"], c["tau0"], c["T"], max(1, c["packets"]),
                      1, sphere=c["ndim"] == 3, vmax_kms=c["vmax"], core_half=c["core"])


def _medium(c, seed):
    """The turbulent lognormal medium at cell resolution; another seed is another medium."""
    return W.clumpy_medium(n=c["cells"], J=c["bins"], x_max=c["xmax"], tau0=c["tau0"], brick=1,
                           seed=0x5EED0005 + int(seed))


def _problem(c, seed):
    if c["clumpy"]:
        return R.Problem.clumpy(_medium(c, seed))
    return R.Problem(_workload(c), mode=R.MODE_HYBRID if c["hybrid"] else R.MODE_DDMC, dust_abs=c["dust"],
                     dust_weights=c["weights"])


def _n_out(c):
    nA, nC = 6 * c["bins"], 6 * c["side"] ** 2
    return nA, nC, (nA + L.N_STEP_BUCKETS + nC + 15) // 16 * 16


def _network(c, seed):
    """Weights (He), inputs in the featurisation's range and targets of one minibatch."""
    nA, nC, n_out = _n_out(c)
    B, S = c["rows"], c["side"] ** 2
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    flat = []
    for o, i in ((128, 16), (128, 128), (128, 128), (n_out, 128)):
        flat += [torch.randn(o * i, device="cuda", generator=g) * math.sqrt(2.0 / i), torch.zeros(o, device="cuda")]
    wf = torch.cat(flat)
    wb = torch.empty_like(wf, dtype=torch.bfloat16)
    R.mlp_to_bf16(n_out, wf.data_ptr(), wb.data_ptr(), torch.cuda.current_stream().cuda_stream)
    x = (2.0 * torch.rand((B, 16), device="cuda", generator=g) - 1.0).to(torch.bfloat16)
    ri = lambda hi: torch.randint(0, hi, (B,), device="cuda", generator=g, dtype=torch.int32)  # noqa: E731
    face = ri(6)
    capped = torch.rand(B, device="cuda", generator=g) < 0.01   # passages cut by the step cap carry no target
    ta = torch.where(capped, -1, face * c["bins"] + ri(c["bins"])).to(torch.int32)
    tc = torch.where(capped, -1, face * S + ri(S)).to(torch.int32)
    return dict(wf=wf, wb=wb, x=x, ta=ta, tb=ri(L.N_STEP_BUCKETS), tc=tc)


def prepare(case, seed):
    c = dict(case)
    k, st = c["kind"], dict(case=c, seed=_philox_seed(seed))
    if k in ("run", "slices"):
        st["p"] = _problem(c, seed)
        st["p"].ensure_state(c["packets"])
    elif k == "time":
        st["p"] = _problem(c, seed)
        st["edges"] = W.time_edges(c["dt"], c["dt"] * c["steps"])
    elif k == "batch":
        ws = W.batched_instances(c["instances"], packet_scale=c["scale"])
        st["stream"] = torch.cuda.Stream()      # a graph is captured on a stream of its own
        with torch.cuda.stream(st["stream"]):
            st["b"] = R.Batch([R.Problem(w) for w in ws], [w.packets for w in ws])
            st["g"] = st["b"].graph(R.RunOpts(st["seed"], 0, c["steps"]))
    elif k == "network":
        st.update(_network(c, seed))
        n_out = _n_out(c)[2]
        st["work"] = torch.empty(R.mlp_work_bytes(c["rows"], n_out), dtype=torch.uint8, device="cuda")
        if c["train"]:
            st["grad"], st["m"], st["v"] = (torch.zeros_like(st["wf"]) for _ in range(3))
            st["loss"], st["step"] = torch.zeros(1, device="cuda"), 0
        else:
            st["logits"] = torch.empty((c["rows"], n_out), device="cuda")
    elif k == "passages":
        med = _medium(c, seed)
        st["prop"] = L.RegionProposal(R.Problem.clumpy(med), med.n_rel, med.v_kms, c["brick"], c["margin"])
    else:
        st["med"] = _medium(c, seed)
    return st


# ----------------------------------------------------------------------------- one pass
def _tallies(t, weights=False):
    keep = ["emitted", "escaped", "aborted", "steps", "mc_events", "conversions", "clamps", "event_draws", "absorbed",
            "hist", "faces", "sb"] + (["escaped_weight", "weight_hist"] if weights else [])
    return {k: t[k] for k in keep}


def run(state):
    c, seed = state["case"], state["seed"]
    k, n = c["kind"], c["packets"]
    if k == "run":
        return _tallies(state["p"].run(n, seed), c["weights"])
    if k == "slices":
        p = state["p"]
        p.reset()
        p.launch(n, seed, steps_per_launch=c["steps"])
        p.launch(n, seed, steps_per_launch=c["steps"], resume=1)
        return dict(tallies=_tallies(p.read()), states=p.packet_states(n, 0, min(n, SAMPLE)))
    if k == "time":
        r = state["p"].time_run(n, seed, state["edges"], leaks=c["leaks"])
        out = {q: r[q] for q in ("bins", "path_ticks", "path", "esc", "dwells", "transitions", "alive")}
        if c["leaks"]:
            out["leak"] = r["leak"]
        return dict(out, tallies=_tallies(r["tallies"]))
    if k == "batch":
        with torch.cuda.stream(state["stream"]):
            state["b"].graph_launch(state["g"])
        return state["b"].tally
    if k == "network":
        nA, nC, n_out = _n_out(c)
        d = {q: v.data_ptr() for q, v in state.items() if isinstance(v, torch.Tensor)}
        s = torch.cuda.current_stream().cuda_stream
        if not c["train"]:
            R.mlp_forward(n_out, d["wf"], d["wb"], d["x"], c["rows"], d["work"], d["logits"], s)
            return state["logits"]
        R.mlp_loss_grad(n_out, nA, L.N_STEP_BUCKETS, d["wf"], d["wb"], d["x"], d["ta"], d["tb"], c["rows"], d["work"],
                        d["grad"], d["loss"], s, nC=nC, S=c["side"] ** 2, d_tc=d["tc"])
        state["step"] += 1
        R.mlp_adam(n_out, d["wf"], d["wb"], d["grad"], d["m"], d["v"], state["step"], 1.0e-3, stream=s)
        return dict(loss=state["loss"], grad=state["grad"])
    if k == "passages":
        return state["prop"].generate(n, seed)
    p = R.Problem.clumpy(state["med"], mode=R.MODE_HYBRID)
    redist = p.redistribution()
    p.reset()
    p.launch(n, seed, steps_per_launch=c["steps"], redist=redist)
    return dict(tallies=_tallies(p.read()), redist=redist,
                tau=R.cell_tau(p.grid, p.table.data_ptr(), 0, p.J, p.stream()))


# ----------------------------------------------------------------------------- necessary work
def work(case):
    """Bytes: inputs read once and outputs written once (rows of the leakage
    table that the states need, packet states in and out, tallies).  Operations:
    OPS per transition, the products of the network, and for a table the
    profile's integrals (about 300 operations each)."""
    c = case
    k, J = c["kind"], c["bins"]
    cells = c["cells"] ** c["ndim"]
    row = 16 if c["ndim"] == 1 else 32
    rows = cells * J if c["clumpy"] else (3 if c["ndim"] == 1 else 27) * J
    if k == "network":
        n_out, B = _n_out(c)[2], c["rows"]
        par = 128 * 16 + 2 * 128 * 128 + 128 * n_out + 3 * 128 + n_out
        mac = B * (128 * 16 + 2 * 128 * 128 + 128 * n_out)
        if not c["train"]:
            return dict(bytes=2 * par + 32 * B + 4 * B * n_out, flops=2 * mac)
        return dict(bytes=(2 + 4 + 4 + 8 + 8 + 4 + 2) * par + 44 * B, flops=6 * mac)
    flops = OPS * c["transitions"]
    if k == "run":
        return dict(bytes=rows * row + 8 * (3 * J), flops=flops)
    if k == "slices":
        return dict(bytes=rows * row + 3 * 25 * c["packets"], flops=flops)
    if k == "time":
        return dict(bytes=c["steps"] * (rows * row + 2 * 33 * c["packets"] + 16 * cells * J), flops=2 * flops)
    if k == "batch":
        return dict(bytes=c["instances"] * 2.0e4, flops=flops)
    if k == "passages":
        return dict(bytes=rows * row + (32 + 8 + 32 + 12) * c["packets"], flops=flops)
    return dict(bytes=rows * row + 32 * cells + 4 * J * (J - 1) + 25 * c["packets"],
                flops=flops + 300 * (3 * cells * (J + 1) + 3 * J * 28 * 16 * 30 * 8))


# ----------------------------------------------------------------------------- 64-bit values
def _layers(c, s):
    """The network's matrices (as rounded to BF16) and biases (FP32) in 64 bits."""
    n_out = _n_out(c)[2]
    o, out = 0, []
    for q, i in ((128, 16), (128, 128), (128, 128), (n_out, 128)):
        out.append((s["wb"][o:o + q * i].double().view(q, i), s["wf"][o + q * i:o + q * i + q].double()))
        o += q * i + q
    return out


def exact(case, seed):
    """The network in 64 bits; every other output is a count, a position or an
    integer number of ticks."""
    c = dict(case)
    if c["kind"] != "network":
        return None
    s = _network(c, seed)
    ws = _layers(c, s)
    h = [s["x"].double()]
    for w, b in ws[:3]:
        h.append(torch.relu(h[-1] @ w.T + b))
    z = h[-1] @ ws[3][0].T + ws[3][1]
    if not c["train"]:
        return z
    nA, nC, n_out = _n_out(c)
    B, S, nB = c["rows"], c["side"] ** 2, L.N_STEP_BUCKETS
    live = s["ta"] >= 0
    ar = torch.arange(B, device="cuda")
    dz, loss = torch.zeros_like(z), torch.zeros(1, dtype=torch.float64, device="cuda")

    def head(lo, width, tgt, z_):
        """Cross-entropy over `width` logits from column lo (a number, or one per row), target tgt in them."""
        cols = (lo if torch.is_tensor(lo) else torch.full((B,), lo, device="cuda"))[:, None].long() + \
            torch.arange(width, device="cuda")[None, :]
        lp = torch.log_softmax(z_.gather(1, cols), 1)
        pr = lp.exp()
        t = tgt.clamp(min=0).long()
        pr[ar, t] -= 1.0
        dz.scatter_(1, cols, pr * live[:, None] / B)
        return -(lp[ar, t] * live).sum()

    loss += head(0, nA, s["ta"], z) + head(nA, nB, s["tb"], z)
    tc = s["tc"].clamp(min=0)
    loss += head(nA + nB + tc // S * S, S, tc % S, z)
    grads = [None] * 4
    d = dz
    for q in (3, 2, 1, 0):
        grads[q] = torch.cat([(d.T @ h[q]).reshape(-1), d.sum(0)])
        if q:
            d = (d @ ws[q][0]) * (h[q] > 0)
    return dict(loss=loss, grad=torch.cat(grads))
