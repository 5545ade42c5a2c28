"""The work that users of the package have it do, as cases that can be timed.

A case is a dict of plain values.  ``kind`` says which entry points it calls:

  sweep     ising_sweep of one lattice (either layout), n sweeps per call
  slabs     ising_slab_sweep of one lattice held as horizontal slabs
  batch     Batch.run: many lattices, recorded and with replica exchange
  host      one sweep of a lattice held in pinned host memory
  snapshot  init, conversions between the layouts and observables
  forward   ising_net_forward, inference
  train     one training step: forward, loss, backward, Adam
  move      BlockMove.move: network, proposal, flipped network, acceptance

Every pass continues from the state that the last one left (sweep indices and
training steps count on), as a running simulation or training does.  Lattices
start from the keyed random state; the network's chains are correlated random
fields cut at zero, which have domains of all sizes as chains near the
critical point do.
"""
import math

import numpy as np
import torch

import paper_1906_06297_gb300 as ising
from paper_1906_06297_gb300.workloads import pt_batch

BETA_C = 0.4406868
CH = 32  # channels of the proposal network


def listed():
    return [
        # the small lattice of a parity or equilibration study: 1000 recorded sweeps in one call, one byte per spin
        {"name": "sweep_int8_256", "kind": "sweep", "layout": "int8", "L": 256, "pad": 0, "n": 1000, "trace": True},
        # the same lattice multi-spin coded, one recorded sweep per call: a program that looks at each state
        {"name": "sweep_msc4_256_once", "kind": "sweep", "layout": "msc4", "L": 256, "pad": 0, "n": 1, "trace": True},
        # a lattice of finite-size studies with ragged rows (66 words) and padding, as in the parity tests
        {"name": "sweep_msc4_2112", "kind": "sweep", "layout": "msc4", "L": 2112, "pad": 32, "n": 20, "trace": True},
        # the smallest lattice of the paper's table for the one-byte layout
        {"name": "sweep_int8_2560", "kind": "sweep", "layout": "int8", "L": 2560, "pad": 0, "n": 10, "trace": False},
        # the benchmark's lattice
        {"name": "sweep_msc4_65536", "kind": "sweep", "layout": "msc4", "L": 65536, "pad": 0, "n": 1, "trace": True},
        # the benchmark's batch: 4096 lattices of sides 32..1024 in 64 ladders, exchange every 10 sweeps
        {"name": "batch_pt", "kind": "batch", "sides": "pt", "ladders": 64, "S": 64, "lo": 0.30, "hi": 0.60, "n": 20, "record": 10},
        # the sampler of the Binder crossing study: sides 64, 128, 256, recorded every second sweep
        {"name": "batch_binder", "kind": "batch", "sides": "64,128,256", "ladders": 8, "S": 16, "lo": 0.42, "hi": 0.46, "n": 100, "record": 2},
        # a lattice kept in pinned host memory, bit-packed, through one sweep
        {"name": "host_bits_32768", "kind": "host", "format": "bits", "L": 32768},
        # a state made, saved in every format and measured
        {"name": "snapshot_16384", "kind": "snapshot", "L": 16384},
        # the proposal network on a side that is no multiple of its row tile
        {"name": "forward_96", "kind": "forward", "L": 96, "C": 256},
        # one training step at the benchmark's minibatch
        {"name": "train_128", "kind": "train", "L": 128, "C": 64},
        # one block move of the benchmark's chains: both evaluations of the network, proposal and acceptance
        {"name": "move_128", "kind": "move", "L": 128, "C": 1024},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "slabs", "batch", "batch", "host", "snapshot", "forward", "train", "move"])
    if kind == "sweep":
        layout = rng.choice(["int8", "msc4"])
        if layout == "int8":
            L = 2 * round(_log(rng, 16, 4096))
            most, pad = 1 << 27, rng.choice([0, 0, rng.randrange(1, 64)])
        else:
            L = 64 * round(_log(rng, 1, 768))
            most, pad = 1 << 32, rng.choice([0, 0, 16 * rng.randrange(1, 8)])
        n = max(1, min(int(_log(rng, 1, 1000)), most // (L * L)))
        return {"kind": kind, "layout": layout, "L": L, "pad": pad, "n": n, "trace": rng.random() < 0.6}
    if kind == "slabs":
        L = 64 * round(_log(rng, 2, 512))
        return {"kind": kind, "L": L, "parts": rng.randrange(1, 6), "n": max(1, min(int(_log(rng, 1, 50)), (1 << 30) // (L * L)))}
    if kind == "batch":
        sides = sorted(rng.sample([32, 64, 96, 128, 160, 192, 256, 384, 512, 640], rng.randrange(1, 4)))
        S = rng.choice([1, 4, 13, 16, 32, 64])
        ladders = max(1, min(int(_log(rng, 1, 64)), (1 << 28) // (S * sum(x * x for x in sides))))
        spins = S * ladders * sum(x * x for x in sides)
        record = rng.choice([0, 1, 2, 5, 10])
        return {"kind": kind, "sides": ",".join(map(str, sides)), "ladders": ladders, "S": S, "lo": 0.42, "hi": 0.46,
                "n": max(1, min(int(_log(rng, 4, 200)), (1 << 32) // spins)), "record": record}
    if kind == "host":
        return {"kind": kind, "format": rng.choice(["bits", "msc4"]), "L": 64 * round(_log(rng, 4, 320))}
    if kind == "snapshot":
        return {"kind": kind, "L": 64 * round(_log(rng, 2, 256))}
    L = 32 * rng.randrange(1, 9)
    area = {"forward": 1 << 24, "train": 1 << 20, "move": 1 << 22}[kind]
    return {"kind": kind, "L": L, "C": max(1, int(_log(rng, 1, area / (L * L))))}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _spins(C, L, seed):
    """C correlated spin fields of side L as 0/1 bytes: white noise averaged over neighbours, cut at zero."""
    f = torch.randn((C, L, L), generator=_generator(seed), device="cuda", dtype=torch.float32)
    for k in range(4):
        d = (1, 2, 3, 1)[k]
        f = f + 0.5 * (torch.roll(f, d, 1) + torch.roll(f, -d, 1))
        f = f + 0.5 * (torch.roll(f, d, 2) + torch.roll(f, -d, 2))
    return (f > 0).to(torch.uint8)


def _planes(s):
    """The MSC4 colour planes (bytes, two spins each) of spins s (C, L, L)."""
    even, odd = s[:, 0::2], s[:, 1::2]
    out = []
    for colour in (0, 1):
        p = torch.empty((s.shape[0], s.shape[1], s.shape[2] // 2), dtype=torch.uint8, device=s.device)
        p[:, 0::2] = even[:, :, colour::2]
        p[:, 1::2] = odd[:, :, 1 - colour::2]
        out.append((p[:, :, 0::2] | (p[:, :, 1::2] << 4)).contiguous())
    return out


def _params(seed):
    """The network's parameters as a training run starts them, with small biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for size, fan_in in ((CH * 9, 9), (CH, 0), (CH * CH * 9, 288), (CH, 0), (CH * CH * 9, 288), (CH, 0), (CH * 9, 288), (1, 0)):
        parts.append(rng.normal(0.0, math.sqrt(2.0 / fan_in) if fan_in else 0.05, size))
    return np.concatenate(parts).astype(np.float32)


def _adam_state(seed, n):
    """First and second moments as after some steps of training."""
    rng = np.random.default_rng(seed + 1)
    return (0.1 * rng.normal(size=n)).astype(np.float32), (0.5 + rng.random(n)).astype(np.float32)


def _batch(case, seed):
    if case["sides"] == "pt":
        L, S, beta = pt_batch(case["ladders"], case["S"], case["lo"], case["hi"])
    else:
        S = case["S"]
        L = [int(x) for x in case["sides"].split(",") for _ in range(case["ladders"] * S)]
        beta = np.linspace(case["lo"], case["hi"], S) if S > 1 else [BETA_C]
    b = ising.Batch(L, S, beta)
    b.init(ising.ISING_INIT_RANDOM, seed)
    return b


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed, "t": 0}
    if kind == "sweep":
        row, _ = ising.ising_lattice_bytes(case["L"], ising.LAYOUTS[case["layout"]])
        st["lat"] = ising.Lattice(case["L"], case["layout"], row_stride_bytes=row + case["pad"])
        if case["pad"]:
            st["lat"].black.zero_()
            st["lat"].white.zero_()
        ising.ising_init_lattice(st["lat"], ising.ISING_INIT_RANDOM, seed)
        st["trace"] = torch.zeros((case["n"], 2), dtype=torch.int64, device="cuda") if case["trace"] else None
    elif kind == "slabs":
        st["slabs"] = [ising.Slab(case["L"], r0, rows) for r0, rows in ising.slab_partition(case["L"], case["parts"])]
        for sl in st["slabs"]:
            ising.ising_slab_init(sl, ising.ISING_INIT_RANDOM, seed)
        st["trace"] = torch.zeros((case["n"], 2), dtype=torch.int64, device="cuda")
    elif kind == "batch":
        st["batch"] = b = _batch(case, seed)
        words = int(b.word_off[-1])
        st["planes"] = [b.ws[o:o + 8 * words] for o in (b._black_off, b._white_off)]
        st["slots"] = [b.ws[o:o + 4 * b.n].view(torch.int32) for o in (b._slot_off, b._at_off)]
    elif kind == "host":
        L = case["L"]
        st["lat"] = ising.Lattice(L, "msc4")
        n = ising.ising_bits_bytes(L)
        ising.ising_init_lattice(st["lat"], ising.ISING_INIT_RANDOM, seed)
        st["stage"] = torch.empty(2 * n, dtype=torch.uint8, device="cuda")
        if case["format"] == "bits":
            ising.ising_msc4_to_bits(st["lat"], st["stage"][:n], st["stage"][n:])
            dev = [st["stage"][:n], st["stage"][n:]]
        else:
            dev = [st["lat"].black, st["lat"].white]
        st["host"] = [torch.empty(d.shape, dtype=torch.uint8, pin_memory=True).copy_(d) for d in dev]
        st["trace"] = torch.zeros((1, 2), dtype=torch.int64, device="cuda")
        st["trace_host"] = torch.zeros((1, 2), dtype=torch.int64).pin_memory()
    elif kind == "snapshot":
        L = case["L"]
        st["lat"], st["back"] = ising.Lattice(L, "msc4"), ising.Lattice(L, "msc4")
        st["bytes"] = ising.Lattice(L, "int8")
        n = ising.ising_bits_bytes(L)
        st["bits"] = [torch.empty(n, dtype=torch.uint8, device="cuda") for _ in range(2)]
        st["obs"] = torch.zeros((2, 2), dtype=torch.int64, device="cuda")
    else:
        L, C = case["L"], case["C"]
        black, white = _planes(_spins(C, L, seed))
        st["params"] = torch.from_numpy(_params(seed)).cuda()
        nb = (L // 8) ** 2
        if kind == "move":
            st["mv"] = mv = ising.BlockMove(L, C, BETA_C)
            mv.black.copy_(black.view(-1))
            mv.white.copy_(white.view(-1))
        else:
            st["black"], st["white"] = black, white
            st["work"] = torch.empty(ising.ising_net_workspace_bytes(L, C, kind == "train"), dtype=torch.uint8, device="cuda")
            st["logits"] = torch.zeros((C, nb), dtype=torch.float32, device="cuda")
        if kind == "train":
            m, v = _adam_state(seed, st["params"].numel())
            st["m"], st["v"] = torch.from_numpy(m).cuda(), torch.from_numpy(v).cuda()
            st["grad"] = torch.zeros_like(st["params"])
            st["dlogits"] = torch.zeros_like(st["logits"])
            st["chain_sq"] = torch.zeros(C, dtype=torch.float32, device="cuda")
            st["loss"] = torch.zeros(1, dtype=torch.float32, device="cuda")
            st["t"] = 100
    return st


def run(st):
    case, seed, t = st["case"], st["seed"], st["t"]
    kind = case["kind"]
    if kind == "sweep":
        lat = st["lat"]
        ising.ising_sweep(lat, BETA_C, case["n"], seed, t, st["trace"])
        st["t"] += case["n"]
        return {"black": lat.black, "white": lat.white, "trace": st["trace"]}
    if kind == "slabs":
        ising.ising_slab_sweep(st["slabs"], BETA_C, case["n"], seed, t, st["trace"])
        st["t"] += case["n"]
        return {"black": [s.black[1:-1] for s in st["slabs"]], "white": [s.white[1:-1] for s in st["slabs"]], "trace": st["trace"]}
    if kind == "batch":
        b = st["batch"]
        events = b.n_events(case["n"], t, case["record"])
        trace = torch.empty((events, b.n, 2), dtype=torch.int64, device="cuda") if events else None
        b.run(case["n"], seed, t, case["record"], case["record"] > 0, trace)
        st["t"] += case["n"]
        return {"planes": st["planes"], "slots": st["slots"], "trace": trace}
    if kind == "host":
        host = st["host"]
        if case["format"] == "bits":
            ising.ising_sweep_host_bits(st["lat"], host[0], host[1], st["stage"], BETA_C, 1, seed, t, st["trace"], st["trace_host"].data_ptr())
        else:
            ising.ising_sweep_host(st["lat"], host[0], host[1], BETA_C, 1, seed, t, st["trace"], st["trace_host"].data_ptr())
        st["t"] += 1
        return {"black": host[0], "white": host[1], "trace": st["trace_host"]}
    if kind == "snapshot":
        lat, by, back, bits, obs = st["lat"], st["bytes"], st["back"], st["bits"], st["obs"]
        ising.ising_init_lattice(lat, ising.ISING_INIT_RANDOM, seed + t)
        ising.ising_observables(lat, obs[0])
        ising.ising_unpack(lat, by)
        ising.ising_observables(by, obs[1])
        ising.ising_msc4_to_bits(lat, bits[0], bits[1])
        ising.ising_pack(by, back)
        ising.ising_bits_to_msc4(bits[0], bits[1], lat)
        st["t"] += 1
        return {"msc4": [lat.black, lat.white], "int8": [by.black, by.white], "bits": bits, "back": [back.black, back.white], "obs": obs}
    L, C = case["L"], case["C"]
    if kind == "forward":
        ising.ising_net_forward(L, C, st["black"], st["white"], None, st["params"], st["logits"], st["work"])
        return {"logits": st["logits"]}
    if kind == "train":
        st["t"] = t = t + 1
        ising.ising_net_forward(L, C, st["black"], st["white"], None, st["params"], st["logits"], st["work"], True)
        ising.ising_net_targets_loss(L, C, st["black"], st["white"], BETA_C, st["logits"], st["dlogits"], st["chain_sq"], st["loss"])
        ising.ising_net_backward(L, C, st["black"], st["white"], st["params"], st["dlogits"], st["grad"], st["work"])
        ising.ising_net_adam(st["params"], st["grad"], st["m"], st["v"], t, 1e-3)
        return {k: st[k] for k in ("logits", "loss", "chain_sq", "dlogits", "grad", "params", "m", "v")}
    mv = st["mv"]
    mv.move(st["params"], seed, t)
    st["t"] += 1
    return {"black": mv.black, "white": mv.white, "logits": mv.lx, "flipped": mv.lxp, "block": mv.block, "accepted": mv.accepted, "dE": mv.dE}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: the inputs once and the outputs once.  Operations: per spin update the 5 wide multiplies of its quarter
    of a Philox4x32-10 block (the neighbour sums and the decision are logic); per pixel of the network 2 per
    multiply-add of the convolutions."""
    kind = case["kind"]
    if kind in ("sweep", "slabs"):
        area = case["L"] ** 2
        per_spin = 1.0 if case.get("layout") == "int8" else 0.5
        return {"bytes": 2 * per_spin * area + 16 * case["n"], "flops": 5.0 * area * case["n"]}
    if kind == "batch":
        if case["sides"] == "pt":
            area = float(sum(x * x for x in pt_batch(case["ladders"], case["S"])[0]))
            count = case["ladders"] * case["S"]
        else:
            sides = [int(x) for x in case["sides"].split(",")]
            area, count = float(case["ladders"] * case["S"] * sum(x * x for x in sides)), case["ladders"] * case["S"] * len(sides)
        events = case["n"] // case["record"] if case["record"] else 0
        return {"bytes": area + 16.0 * count * events, "flops": 5.0 * area * case["n"]}
    area = float(case["L"] ** 2)
    if kind == "host":  # the host's copy and, if it is bit-packed, the device's expanded state
        return {"bytes": (2 / 8 if case["format"] == "bits" else 2 * 0.5) * area, "flops": 5.0 * area}
    if kind == "snapshot":  # each call's input and output
        return {"bytes": (0.5 + 0.5 + (0.5 + 1) + 1 + (0.5 + 0.125) + (1 + 0.5) + (0.125 + 0.5)) * area, "flops": 5.0 * area}
    px = case["C"] * area
    macs = 9 * CH + 2 * 9 * CH * CH + 9 * CH
    n_par = 9 * CH + CH + 2 * (9 * CH * CH + CH) + 9 * CH + 1
    if kind == "forward":
        return {"bytes": 0.5 * px + 4 * px / 64 + 4 * n_par, "flops": 2.0 * macs * px}
    if kind == "train":  # weight gradients of all layers, data gradients of the last three
        return {"bytes": 0.5 * px + 3 * 4 * px / 64 + 4 * n_par * 8, "flops": 2.0 * px * (2 * macs + 2 * 9 * CH * CH + 9 * CH)}
    # a flipped block reaches 4 rows to each side of its 8, through layers of which the first sees 1 row beyond
    return {"bytes": 0.5 * px + 2 * 4 * px / 64 + 4 * n_par, "flops": 2.0 * px * macs * (1 + min(1.0, 26.0 / case["L"]))}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _weights(theta):
    th = torch.from_numpy(theta.astype(np.float64)).cuda()
    out, o = [], 0
    for cin, cout in ((1, CH), (CH, CH), (CH, CH), (CH, 1)):
        n = cin * cout * 9
        out += [th[o:o + n].view(cout, cin, 9).clone().requires_grad_(True), th[o + n:o + n + cout].clone().requires_grad_(True)]
        o += n + cout
    return out


def _net(w, s):
    """Logits (C, blocks) of spins s (C, L, L, +1/-1): 3 x 3 periodic correlations, GELU between, block means."""
    a = s[..., None]
    C, L = s.shape[0], s.shape[1]
    for i in range(4):
        W, b = w[2 * i], w[2 * i + 1]
        z = b.expand(C, L, L, b.numel())
        for k in range(9):
            z = z + torch.roll(a, (1 - k // 3, 1 - k % 3), (1, 2)) @ W[:, :, k].t()
        a = 0.5 * z * (1 + torch.erf(z / math.sqrt(2.0))) if i < 3 else z
    return a[..., 0].view(C, L // 8, 8, L // 8, 8).mean(dim=(2, 4)).reshape(C, -1)


def _block_dE(s):
    """Twice the sum of s_in s_out over the bonds that leave each 8 x 8 block."""
    C, L = s.shape[0], s.shape[1]
    n = L // 8
    right = (s * torch.roll(s, -1, 2)).view(C, n, 8, n, 8)[..., 7].sum(2)   # bonds to the block on the right
    down = (s * torch.roll(s, -1, 1)).view(C, n, 8, n, 8)[:, :, 7].sum(3)  # and below
    return (2 * (right + torch.roll(right, 1, 2) + down + torch.roll(down, 1, 1))).reshape(C, -1)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("forward", "train", "move"):
        return None  # whole numbers
    L, C = case["L"], case["C"]
    s = _spins(C, L, seed).double() * 2 - 1
    theta = _params(seed)
    w = _weights(theta)
    step = max(1, (1 << 20) // (L * L))
    if kind != "train":
        with torch.no_grad():
            logits = torch.cat([_net(w, s[i:i + step]) for i in range(0, C, step)])
        if kind == "forward":
            return {"logits": logits}
        return {"black": None, "white": None, "logits": logits, "flipped": None, "block": None, "accepted": None, "dE": None}
    target = torch.clamp(-BETA_C * _block_dE(s), max=0.0)
    size = target.numel()
    step = max(1, (1 << 19) // (L * L))
    rows = []
    for i in range(0, C, step):
        lo = _net(w, s[i:i + step])
        (((lo - target[i:i + step]) ** 2).sum() / size).backward()
        rows.append(lo.detach())
    logits = torch.cat(rows)
    grad = torch.cat([x.grad.reshape(-1) for x in w])
    m, v = (torch.from_numpy(x.astype(np.float64)).cuda() for x in _adam_state(seed, theta.size))
    t = 101
    m = 0.9 * m + 0.1 * grad
    v = 0.999 * v + 0.001 * grad * grad
    params = torch.from_numpy(theta.astype(np.float64)).cuda()
    params = params - 1e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    r = logits - target
    return {"logits": logits, "loss": (r * r).mean().reshape(1), "chain_sq": (r * r).sum(1), "dlogits": 2 * r / size, "grad": grad,
            "params": params, "m": m, "v": v}
