"""The work that a user of the step library has it do, as cases for timing.

Kinds of case:
  sim      windows of `steps` steps of one network, the raster and the
           message counts read back after each window (the main use: simulate,
           read the spikes); with `tune` the program has run the autotuner
           from the state it simulates from, as the usage notes do;
  batch    the same for independent networks stepped together by one sim;
  loop     closed loop: a few steps, then the membrane state read back, so
           that the caller can react (launch and read-back latency count);
  stim     external stimulation: a caller-given spike pattern routed and
           fanned out into an input buffer;
  setup    a network given as an edge list brought up from nothing:
           partitioned (Algorithm 1 on the GPU), routing tables built on the
           GPU, sim created, a first short run read back;
  adjoint  one training step of the differentiable form through autograd:
           forward, loss on population rates, gradients of gains and drives.

Networks follow the repository's recipe (80 % excitatory, a mix of own
partition / own virtual node / remote targets, int16 weights, delays in
steps); they are drawn on the GPU so that making them is quick.
"""
import math

import numpy as np
import torch

import paper_2205_07125_gb300 as snn

DEV = "cuda:0"
NONE = -1  # an empty place of a record
WINDOWS = 16  # windows of steps that a sim records before it starts again from rest

# ---------------------------------------------------------------- cases


def listed():
    return [
        # the smallest network in use: 4,096 neurons with delay 1 and the library's defaults; every step is
        # latency (launch-free inside the call, two grid-wide exchanges per step)
        {"name": "sim-tiny-4k", "kind": "sim", "M": 4096, "P": 4, "vn": 2, "K": 100, "mix": False, "dmax": 1,
         "steps": 1000, "w_ext": 96, "relabel": False, "tune": False, "delivery": 0, "rest": 0},
        # 1 ms of closed-loop control of a small network: 10 steps and the membrane state per call
        {"name": "loop-16k", "kind": "loop", "M": 16384, "P": 8, "vn": 4, "K": 100, "mix": True, "dmax": 8,
         "steps": 10, "w_ext": 96, "relabel": False, "delivery": 0},
        # a network whose ids say nothing about its partitions (what Algorithm 1 returns for real data): the
        # partition study's size, 65,536 neurons, 200 synapses each
        {"name": "sim-relabelled-65k", "kind": "sim", "M": 65536, "P": 16, "vn": 4, "K": 200, "mix": True, "dmax": 8,
         "steps": 1000, "w_ext": 96, "relabel": True, "tune": False, "delivery": 0, "rest": 200},
        # odd sizes: neurons not a multiple of 4, partitions of unequal size, short delays
        {"name": "sim-ragged-200k", "kind": "sim", "M": 200003, "P": 15, "vn": 5, "K": 137, "mix": True, "dmax": 5,
         "steps": 500, "w_ext": 96, "relabel": False, "tune": False, "delivery": 0, "rest": 200},
        # the scale workload: 1,048,576 neurons, 1,000 synapses each, 64 partitions in 16 virtual nodes, autotuned
        {"name": "sim-scale-1m", "kind": "sim", "M": 1 << 20, "P": 64, "vn": 16, "K": 1000, "mix": True, "dmax": 8,
         "steps": 500, "w_ext": 89, "relabel": False, "tune": True, "delivery": 2, "rest": 1000},
        # the per-GPU share of the paper's run: 5,000,000 neurons in 256 partitions of 64 virtual nodes (neuron
        # state and input far larger than the chip holds), with 200 synapses each so that it is made in seconds
        {"name": "sim-share-5m", "kind": "sim", "M": 5_000_000, "P": 256, "vn": 64, "K": 200, "mix": True, "dmax": 8,
         "steps": 250, "w_ext": 96, "relabel": False, "tune": True, "delivery": 2, "rest": 1000},
        # a batch of independent networks of uneven size, 100 to 1,000 synapses per neuron, stepped together
        {"name": "batch-16", "kind": "batch", "nets": 16, "M_lo": 10_000, "M_hi": 500_000, "K_lo": 100, "K_hi": 1000,
         "steps": 250, "tune": True, "delivery": 2, "rest": 500},
        # a small stimulus: 64 spikes into the 65,536-neuron network
        {"name": "stim-64", "kind": "stim", "M": 65536, "P": 16, "vn": 4, "K": 200, "dmax": 8, "n": 64,
         "relabel": True},
        # a large one: the input that a volley of 20,000 spikes produces in a network of 262,144 neurons
        {"name": "stim-20k", "kind": "stim", "M": 262144, "P": 32, "vn": 8, "K": 500, "dmax": 8, "n": 20000,
         "relabel": False},
        # from an edge list to the first spikes, the partition study's network
        {"name": "setup-65k", "kind": "setup", "M": 65536, "P": 16, "vn": 4, "K": 200, "dmax": 8, "steps": 100,
         "iters": 4},
        # a training step of a small network: 4,096 neurons, 120 steps, checkpoints every 32
        {"name": "adjoint-4k", "kind": "adjoint", "M": 4096, "P": 4, "vn": 2, "K": 64, "dmax": 8, "T": 120,
         "ckpt": 32},
        # a training step of the adjoint workload: 131,072 neurons, 500 synapses each, 500 steps, checkpoints every 50
        {"name": "adjoint-131k", "kind": "adjoint", "M": 131072, "P": 8, "vn": 2, "K": 500, "dmax": 8, "T": 500,
         "ckpt": 50},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sim", "sim", "sim", "sim", "batch", "loop", "stim", "setup", "adjoint", "adjoint"])
    if kind == "batch":
        return {"kind": kind, "nets": rng.randint(4, 24), "M_lo": 10_000, "M_hi": rng.randint(20_000, 120_000),
                "K_lo": 100, "K_hi": rng.randint(200, 1000), "steps": rng.randint(50, 250), "tune": True,
                "delivery": 2, "rest": 200}
    if kind == "adjoint":
        vn = rng.choice([1, 2, 2, 4])
        M = _log(rng, 2000, 120_000)
        T = _log(rng, 40, 400)
        return {"kind": kind, "M": M, "P": vn * rng.randint(2, 4), "vn": vn, "K": rng.randint(40, 450),
                "dmax": rng.choice([1, 4, 8, 8, 12]), "T": T, "ckpt": min(T, rng.randint(10, 100))}
    vn = rng.choice([2, 3, 4, 8])
    P = vn * rng.randint(2, 4)
    M = _log(rng, 4000, 1_000_000) if kind == "sim" else _log(rng, 2000, 100_000)
    K = _log(rng, 50, min(1000, 400_000_000 // M))
    c = {"kind": kind, "M": M, "P": P, "vn": vn, "K": K, "dmax": rng.choice([1, 2, 5, 8, 8, 8]),
         "relabel": rng.random() < 0.5}
    if kind == "sim":
        # networks of 1 to 16 steps of delay, the defaults or an autotuned sim, any delivery that the size allows
        tune = rng.random() < 0.5
        c.update(mix=rng.random() < 0.75, steps=rng.randint(50, 400), w_ext=89 if K > 300 else 96, tune=tune,
                 delivery=2 if tune else rng.choice([0, 0, 1, 2]), rest=rng.choice([0, 200]))
        if not tune and c["delivery"] == 0 and rng.random() < 0.2:
            c["dmax"] = 16
    elif kind == "loop":
        c.update(mix=True, steps=rng.randint(1, 20), w_ext=96, delivery=rng.choice([0, 0, 2]))
    elif kind == "stim":
        c.update(n=_log(rng, 1, min(M, 20_000)))
    else:
        c.update(steps=rng.randint(20, 150), iters=rng.randint(1, 4))
        del c["relabel"]
    return c


# ---------------------------------------------------------------- networks
def _starts(M, P):
    return (np.arange(P + 1, dtype=np.int64) * M) // P


def _mix(K):
    n_part = int(round(0.7 * K))
    n_vn = int(round(0.2 * K))
    return n_part, n_vn, K - n_part - n_vn


def _fill(g, M, P, vn, K, mix, dmax, tgt, w, d, perm):
    """Targets, weights and delays of one network into the [M, K] arrays tgt, w, d (host), ids relabelled by perm."""
    st = torch.from_numpy(_starts(M, P)).to(DEV)
    vs = P // vn
    n_part, n_vn, n_rem = _mix(K)
    if vn == 1:
        n_vn, n_rem = n_vn + n_rem, 0
    rows = max(1, (1 << 26) // K)
    inv = None if perm is None else torch.argsort(perm)

    def below(n, cols):
        r = torch.randint(0, 1 << 31, (n.shape[0], cols), generator=g, device=DEV)
        return (r * n[:, None]) >> 31

    for a in range(0, M, rows):
        b = min(M, a + rows)
        # row r of the arrays is neuron r; its place in the planted order is i
        i = torch.arange(a, b, device=DEV) if inv is None else inv[a:b]
        p = torch.bucketize(i, st, right=True) - 1
        ps, pe = st[p], st[p + 1]
        if not mix:
            t = below(torch.full_like(i, M - 1), K)
            t += t >= i[:, None]
        else:
            v0, v1 = st[p // vs * vs], st[(p // vs + 1) * vs]
            own = below(pe - ps - 1, n_part) + ps[:, None]
            own += own >= i[:, None]
            peer = below(v1 - v0 - (pe - ps), n_vn) + v0[:, None]
            peer += (peer >= ps[:, None]) * (pe - ps)[:, None]
            far = below(M - (v1 - v0), n_rem)
            far += (far >= v0[:, None]) * (v1 - v0)[:, None]
            t = torch.cat([own, peer, far], 1)
        if perm is not None:
            t = perm[t]
        exc = ((i - ps) < torch.floor(0.8 * (pe - ps) + 0.5))[:, None]
        z = torch.randn((b - a, K), generator=g, device=DEV)
        ww = torch.where(exc, torch.clamp(torch.round(40 + 8 * z), 1, 32767),
                         -torch.clamp(torch.round(160 + 32 * z), 1, 32768))
        dd = torch.randint(1, dmax + 1, (b - a, K), generator=g, device=DEV, dtype=torch.int32)
        torch.from_numpy(tgt[a:b]).copy_(t.to(torch.int32))
        torch.from_numpy(w[a:b]).copy_(ww.to(torch.int16))
        torch.from_numpy(d[a:b]).copy_(dd.to(torch.uint8))


class _Net:
    """A network's arrays (host), its partition labels and its excitatory flags."""

    def __init__(self, M, P, vn, K, mix, dmax, relabel, seed):
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        self.M, self.K, self.P, self.vn = M, K, P, vn
        perm = torch.randperm(M, generator=g, device=DEV) if relabel else None
        self.tgt = np.empty((M, K), np.int32)
        self.w = np.empty((M, K), np.int16)
        self.d = np.empty((M, K), np.uint8)
        _fill(g, M, P, vn, K, mix, dmax, self.tgt, self.w, self.d, perm)
        self.v0 = (-65.0 + 15.0 * torch.rand(M, generator=g, device=DEV)).cpu().numpy()
        st = _starts(M, P)
        part = np.repeat(np.arange(P, dtype=np.int32), np.diff(st))
        exc = (np.arange(M) - st[part]) < np.floor(0.8 * np.diff(st)[part] + 0.5)
        if perm is not None:
            inv = torch.argsort(perm).cpu().numpy()
            part, exc = part[inv], exc[inv]
        self.part, self.is_exc = np.ascontiguousarray(part), np.ascontiguousarray(exc, np.uint8)

    def network(self):
        return snn.Network(np.arange(self.M + 1, dtype=np.int64) * self.K, self.tgt.reshape(-1).view(np.uint32),
                           self.w.reshape(-1), self.d.reshape(-1), self.v0)


def _net(c, seed):
    return _Net(c["M"], c["P"], c["vn"], c["K"], c.get("mix", True), c["dmax"], c.get("relabel", False), seed)


class _Dyn:
    dt_ms, tau_ms, e_l, v_th, v_reset, t_ref = 0.1, 20.0, -65.0, -50.0, -65.0, 20
    i_bias = 0

    def __init__(self, w_ext, seed, lam=0.8):
        self.w_ext, self.drive_seed, self.drive_lambda = w_ext, 2000 + seed, lam


def _params(c, dyn, M):
    # raster room for 30 Hz (0.003 spikes per neuron and step) and a volley of every neuron
    if c["kind"] == "loop":  # the caller reads the state, nothing is recorded
        return snn.sim_params(dyn, delivery=c["delivery"])
    n = WINDOWS * c["steps"]
    return snn.sim_params(dyn, delivery=c["delivery"], raster_steps=n + 1500, raster_cap=int(0.003 * M * n) + 4 * M)


def _batch(c, seed):
    """Networks concatenated: sizes log-uniform, out-degrees and drives uniform, 4 to 32 partitions in VNs of 2."""
    r = np.random.default_rng(c["nets"])  # the batch's composition is the case's, its synapses the seed's
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    sizes = [int(np.exp(r.uniform(np.log(c["M_lo"]), np.log(c["M_hi"])))) // 4 * 4 for _ in range(c["nets"])]
    ks = [int(r.integers(c["K_lo"], c["K_hi"] + 1)) for _ in sizes]
    ps = [2 * int(r.integers(2, 17)) for _ in sizes]
    rates = [float(r.uniform(5, 15)) for _ in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    poff = np.concatenate([[0], np.cumsum(ps)])
    M = int(off[-1])
    ptr = np.concatenate([[0], np.cumsum(np.repeat(ks, sizes))]).astype(np.int64)
    tgt, w, d = np.empty(ptr[-1], np.int32), np.empty(ptr[-1], np.int16), np.empty(ptr[-1], np.uint8)
    part = np.empty(M, np.int32)
    for k, m in enumerate(sizes):
        a, b = ptr[off[k]], ptr[off[k + 1]]
        _fill(g, m, ps[k], ps[k] // 2, ks[k], True, 8, tgt[a:b].reshape(m, -1), w[a:b].reshape(m, -1),
              d[a:b].reshape(m, -1), None)
        tgt[a:b] += np.int32(off[k])
        part[off[k]:off[k + 1]] = poff[k] + np.repeat(np.arange(ps[k], dtype=np.int32), np.diff(_starts(m, ps[k])))
    v0 = (-65.0 + 15.0 * torch.rand(M, generator=g, device=DEV)).cpu().numpy()
    net = snn.Network(ptr, tgt.view(np.uint32), w, d, v0)
    rt = snn.Routing(net, part, int(poff[-1]), int(poff[-1]) // 2, "contiguous", build="device", device=DEV)
    plist = [_params(c, _Dyn(89, 100 * seed + k, 0.8 * rates[k] / 10), M) for k in range(len(sizes))]
    return snn.Sim(net, rt, plist[0], device=DEV, batch=(off, plist))


# ---------------------------------------------------------------- what the user has in hand, and a pass
class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, kind, M = case, case["kind"], case.get("M", 0)
    if kind in ("sim", "loop"):
        n = _net(case, seed)
        net = n.network()
        rt = snn.Routing(net, n.part, n.P, n.vn, "contiguous", build="device", device=DEV)
        s.sim = snn.Sim(net, rt, _params(case, _Dyn(case["w_ext"], seed), n.M), device=DEV)
    elif kind == "batch":
        s.sim = _batch(case, seed)
        M = s.sim.M
    elif kind == "stim":
        n = _net(case, seed)
        net = n.network()
        rt = snn.Routing(net, n.part, n.P, n.vn, "contiguous", build="device", device=DEV)
        s.sim = snn.Sim(net, rt, snn.sim_params(_Dyn(96, seed)), device=DEV)
        g = torch.Generator(device=DEV)
        g.manual_seed(seed + 1)
        s.ids = torch.randint(0, n.M, (case["n"],), generator=g, device=DEV, dtype=torch.int32)
        s.out = torch.empty((case["dmax"], n.M), dtype=torch.int32, device=DEV)
    elif kind == "setup":
        n = _Net(case["M"], case["P"], case["vn"], case["K"], True, case["dmax"], True, seed)
        s.net, s.seed = n.network(), seed
    else:
        n = _net(case, seed)
        net = n.network()
        rt = snn.Routing(net, n.part, n.P, n.vn, "contiguous", build="device", device=DEV)
        s.adj = snn.Adjoint(net, n.is_exc, rt, snn.sim_params(_Dyn(89, seed), raster_cap=0),
                            snn.adjoint_params(T=case["T"], ckpt_every=case["ckpt"]), device=DEV)
        G, lam, s.target = (x.to(DEV) for x in _gains(case, seed))
        s.G, s.lam = G.requires_grad_(), lam.requires_grad_()
        s.f = snn.make_adjoint_function()
    if kind in ("sim", "batch", "setup"):
        # the program's own record of a window: ids, then the mark of an empty place
        s.ids, s.n = np.full(int(0.003 * M * case["steps"]) + M, NONE, np.int32), 0
    if kind in ("sim", "batch"):
        s.t = case["rest"]
        if case["rest"]:
            s.sim.step(case["rest"])  # past the transient from rest
        if case["tune"]:
            s.sim.autotune(60)
    return s


def _gains(case, seed):
    """Population-pair gains around 1, drives around 0.85 arrivals per step, target rates of 5 to 15 Hz."""
    g = torch.Generator()
    g.manual_seed(seed + 2)
    n_pop = 2 * case["vn"]
    return (1.0 + 0.25 * torch.randn((n_pop, n_pop), generator=g), 0.7 + 0.3 * torch.rand(n_pop, generator=g),
            (0.0005 + 0.001 * torch.rand(n_pop, generator=g)).double())


def _keep(s, sim, t0, t1):
    """Reads the spikes of steps t0 .. t1-1 into the program's record."""
    ids, off = sim.read_raster(t0, t1)
    s.ids[:len(ids)] = ids
    s.ids[len(ids):s.n] = NONE
    s.n = len(ids)
    return off


def run(s):
    c = s.case
    kind = c["kind"]
    if kind in ("sim", "batch"):
        T = c["steps"]
        if s.t + T > WINDOWS * T + 1500:
            s.sim.reset()
            s.t = 0
        s.sim.step(T)
        off = _keep(s, s.sim, s.t, s.t + T)
        s.t += T
        return {"ids": s.ids, "off": off, "counts": s.sim.read_counts()}
    if kind == "loop":
        s.sim.step(c["steps"])
        V, ref, t = s.sim.read_state()
        return {"V": V, "ref": ref, "t": t}
    if kind == "stim":
        s.out.zero_()
        return {"counts": s.sim.deliver_spikes(s.ids, s.out), "out": s.out}
    if kind == "setup":
        part, stats = snn.snn_partition_device(s.net, c["P"], iters=c["iters"], seed=7 + s.seed, device=DEV)
        rt = snn.Routing(s.net, part, c["P"], c["vn"], "greedy", build="device", device=DEV)
        prm = snn.sim_params(_Dyn(96, s.seed), raster_steps=c["steps"], raster_cap=int(0.003 * c["M"] * c["steps"]) + c["M"])
        sim = snn.Sim(s.net, rt, prm, device=DEV)
        sim.step(c["steps"])
        off = _keep(s, sim, 0, c["steps"])
        out = {"part": part, "stats": stats, "groups": rt.groups()[0], "ids": s.ids, "off": off,
               "counts": sim.read_counts()}
        sim.close()
        rt.close()
        return out
    s.G.grad = s.lam.grad = None
    rates = s.f.apply(s.G, s.lam, s.adj)
    loss = ((rates - s.target) ** 2).mean()
    loss.backward()
    return {"rates": rates.detach(), "loss": loss.detach(), "dG": s.G.grad, "dlam": s.lam.grad}


# ---------------------------------------------------------------- what a pass cannot do without
RATE = 1e-3  # spikes per neuron and step near the networks' working point (10 Hz)


def work(case):
    """Bytes: the synapses (6 B) and routing entries (16 B per destination partition) of the spikes, the neuron state
    (V, refractory counter) and what comes back, each once per pass; flops: the float operations of the neuron updates
    (6 per neuron and step) and of the gradient terms (2 per synapse and step)."""
    kind = case["kind"]
    if kind == "batch":
        M = case["nets"] * (case["M_hi"] - case["M_lo"]) / math.log(case["M_hi"] / case["M_lo"])
        K = (case["K_lo"] + case["K_hi"]) / 2
        seg = min(18, K)
    else:
        M, K = case["M"], case["K"]
        seg = min(case["P"], K)
    per_spike = 6 * K + 16 * seg
    if kind == "stim":
        return {"bytes": case["n"] * (4 + per_spike) + 4 * case["dmax"] * M, "flops": 0}
    if kind == "adjoint":
        T, E = case["T"], M * K
        # forward: the spikes' synapses; backward: every synapse once per pass at least, the recorded state per step
        return {"bytes": 2 * T * RATE * M * per_spike + 6 * E + 10 * M, "flops": 2 * T * 8 * M + 2 * T * E}
    T = case["steps"]
    b = 10 * M + T * RATE * M * (per_spike + 4)
    if kind == "setup":
        b += 7 * M * K * 2 + 4 * M  # the edge list read for the partition and for the tables
    return {"bytes": b, "flops": 6 * T * M}


# ---------------------------------------------------------------- 64-bit values
M32 = 0xFFFFFFFF


def _mulhilo(a, b):
    """High and low words of the 32 x 32 bit product (a: int64 tensor of 32-bit values, b: constant)."""
    b0, b1 = b & 0xFFFF, b >> 16
    p0, p1 = a * b0, a * b1              # below 2^48 each
    s = p0 + ((p1 & 0xFFFF) << 16)       # below 2^49
    return (p1 >> 16) + (s >> 32), s & M32


def _philox(key, c0, c1, c2):
    """Philox4x32-10 (Salmon et al., SC'11) of counter (c0, c1, c2, 0): four words as int64 tensors."""
    k0, k1 = key & M32, key >> 32
    x0, x1, x2, x3 = c0, torch.full_like(c0, c1), torch.full_like(c0, c2), torch.zeros_like(c0)
    for _ in range(10):
        h0, l0 = _mulhilo(x0, 0xD2511F53)
        h1, l1 = _mulhilo(x2, 0xCD9E8D57)
        x0, x1, x2, x3 = h1 ^ x1 ^ k0, l1, h0 ^ x3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x0, x1, x2, x3


def exact(case, seed):
    if case["kind"] == "loop":
        return _exact_loop(case, seed)
    if case["kind"] == "adjoint" and case["M"] * case["K"] * case["T"] <= 4.0e10:
        return _exact_adjoint(case, seed)
    return None  # whole numbers


def _exact_loop(c, seed):
    """The first pass from rest, in 64 bits."""
    n, dyn = _net(c, seed), _Dyn(c["w_ext"], seed)
    M = n.M
    V, ref = n.v0.astype(np.float64), np.zeros(M, np.int64)
    ring = np.zeros((c["dmax"] + 1, M), np.int64)
    cdf, pmf, th = 0.0, math.exp(-dyn.drive_lambda), []
    for k in range(32):
        pmf = pmf if k == 0 else pmf * dyn.drive_lambda / k
        cdf += pmf
        x = math.floor(cdf * 2.0 ** 32)
        if x >= 2 ** 32 - 1:
            break
        th.append(x)
    alpha = math.exp(-dyn.dt_ms / dyn.tau_ms)
    for t in range(c["steps"]):
        quads = torch.arange((M + 3) // 4)
        words = torch.stack(_philox(dyn.drive_seed, quads, t, 0), 1).reshape(-1)[:M].numpy()
        k = np.searchsorted(np.array(th), words, side="right")
        slot = t % (c["dmax"] + 1)
        I = ring[slot] + k * dyn.w_ext
        ring[slot] = 0
        live = ref == 0
        V = np.where(live, dyn.e_l + alpha * (V - dyn.e_l) + I / 1024.0, dyn.v_reset)
        spk = live & (V >= dyn.v_th)
        ref = np.where(spk, dyn.t_ref, np.maximum(ref - 1, 0))
        V[spk] = dyn.v_reset
        for i in np.nonzero(spk)[0]:
            np.add.at(ring, ((t + n.d[i].astype(np.int64)) % (c["dmax"] + 1), n.tgt[i]), n.w[i].astype(np.int64))
    return {"V": V, "ref": None, "t": None}


def _exact_adjoint(c, seed):
    """Rates, loss and gradients of the training step in 64 bits on the trajectory of the 32-bit forward (the spikes
    are part of the inputs of the backward pass: a threshold decision has no 64-bit value)."""
    n, dyn = _net(c, seed), _Dyn(89, seed)
    M, K, T, D, NP = n.M, n.K, c["T"], c["dmax"] + 1, 2 * c["vn"]
    tgt = torch.from_numpy(n.tgt).to(DEV)
    w = torch.from_numpy(n.w).to(DEV)
    d = torch.from_numpy(n.d).to(DEV)
    pop_h = 2 * (n.part // (n.P // n.vn)) + 1 - n.is_exc.astype(np.int64)
    pop = torch.from_numpy(pop_h.astype(np.int64)).to(DEV)
    G, lam, target = (x.to(DEV) for x in _gains(c, seed))
    f32 = torch.float32
    alpha = torch.tensor(math.exp(-dyn.dt_ms / dyn.tau_ms), dtype=f32, device=DEV)
    V = torch.from_numpy(n.v0).to(DEV)
    ref = torch.zeros(M, dtype=torch.int32, device=DEV)
    ring = torch.zeros((D, M, NP), dtype=torch.int32, device=DEV)
    ids = torch.arange(M, device=DEV)
    vpre = torch.empty((T, M), dtype=f32, device=DEV)
    spk = torch.empty((T, M), dtype=torch.bool, device=DEV)
    live = torch.empty((T, M), dtype=torch.bool, device=DEV)
    A = torch.empty((T, M, NP), dtype=torch.int32, device=DEV)
    cnt = torch.zeros(NP, dtype=torch.int64, device=DEV)
    for t in range(T):
        a = ring[t % D]
        A[t] = a
        af = a.to(f32)
        irec = G[pop, 0] * af[:, 0]
        for b in range(1, NP):
            irec = irec + G[pop, b] * af[:, b]
        words = _philox(dyn.drive_seed, ids, t, 0xAD)
        noise = sum((x >> s) & 0xFF for x in words[:3] for s in (0, 8, 16, 24)) - 1530
        xi = noise.to(f32) / 256.0
        I = irec + float(dyn.w_ext) * (lam[pop] + torch.tensor(0.9, dtype=f32, device=DEV) * xi)
        u = V - dyn.e_l
        vp = dyn.e_l + alpha * u
        vp = vp + I * 0.0009765625
        l = ref == 0
        s = l & (vp >= dyn.v_th)
        vpre[t], spk[t], live[t] = vp, s, l
        V = torch.where(l & ~s, vp, torch.full_like(vp, dyn.v_reset))
        ref = torch.where(s, torch.full_like(ref, dyn.t_ref), torch.clamp(ref - 1, min=0))
        ring[t % D] = 0
        i = torch.nonzero(s).reshape(-1)
        if i.numel():
            cnt += torch.bincount(pop[i], minlength=NP)
            at = (((t + d[i].long()) % D) * M + tgt[i].long()) * NP + pop[i][:, None]
            ring.view(-1).index_add_(0, at.reshape(-1), w[i].to(torch.int32).reshape(-1))
    size = torch.bincount(pop, minlength=NP).double()
    rates = cnt.double() / (T * size)
    G64, c10 = G.double(), 2.0 ** -10
    direct = 2.0 * (rates - target) / NP / (T * size)
    gv = torch.zeros(M, dtype=torch.float64, device=DEV)
    H = torch.zeros((D, NP, M), dtype=torch.float64, device=DEV)  # G[pop k][b] * adjoint of k at step t, slot t mod D
    dG = torch.zeros((NP, NP), dtype=torch.float64, device=DEV)
    dl = torch.zeros(NP, dtype=torch.float64, device=DEV)
    rows = max(1, (1 << 26) // K)
    base = pop * M
    total = torch.empty(M, dtype=torch.float64, device=DEV)
    for t in range(T - 1, -1, -1):
        for r in range(0, M, rows):
            e = min(M, r + rows)
            at = ((t + d[r:e].long()) % D) * (NP * M) + base[r:e, None] + tgt[r:e]
            total[r:e] = (H.view(-1)[at] * w[r:e]).sum(1)
        gs = direct[pop] + c10 * total
        sg = 1.0 / (1.0 + 5.0 * (vpre[t].double() - dyn.v_th).abs()) ** 2
        gvp = torch.where(live[t], torch.where(spk[t], torch.zeros_like(gv), gv) + gs * sg, torch.zeros_like(gv))
        H[t % D] = G64.t()[:, pop] * gvp
        gv = alpha.double() * gvp
        dG.index_add_(0, pop, (gvp * c10)[:, None] * A[t].double())
        dl.index_add_(0, pop, gvp * c10 * dyn.w_ext)
    loss = ((rates - target) ** 2).mean()
    return {"rates": rates, "loss": loss, "dG": dG, "dlam": dl}
