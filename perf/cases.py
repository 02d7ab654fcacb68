"""The work whose speed counts: calls of the public entry points over the sizes, signatures and options that users have.

listed() is a fixed selection, draw() gives further cases of the same ranges.  A case names one kind of call:

  conv        e3j_conv_fwd and / or e3j_conv_bwd over a prepared neighbour list (the message-passing layer)
  padded      the same for a batch whose edge list is padded to a fixed capacity, the list prepared in the call
  md          a molecular-dynamics step: e3j_graph_prepare for the new list, forward and backward on edge vectors
  radial      forward and backward on edge vectors with the weights given by the radial network's last layer (h, W)
  training    forward, backward and double backward (a loss on forces)
  tp          the standalone channelwise tensor product, forward and backward
  f64         forward and backward in float64

Graphs are periodic boxes of atoms drawn from the seed (water, a liquid of single atoms, water of uneven density, plain
points), cut at the radius that gives the stated number of neighbours, so that a case has the same number of edges
whatever the seed.  Features, weights and cotangents are N(0, 1); W is N(0, 1 / hidden), so that h W has unit scale.
"""
import math

import numpy as np
import torch

import paper_2609_35099_b200 as e3j
from paper_2609_35099_b200 import workloads

WATER, HIGHORDER, TP = "128x0e+128x1o", "64x0e+64x1o+64x2e+64x3o", "128x0e+128x1o+128x2e"


def listed():
    return [
        # A small cluster and few channels: what a unit test or a toy potential calls; launches and latency.
        dict(name="tiny", kind="conv", passes="both", irreps="8x0e+8x1o", lmax=2, out="0e+1o+1e+2e+2o", system="points",
             atoms=64, neighbours=32),
        # A batch of small molecules in a fixed-capacity edge list, outputs of natural parity; the list is new each time.
        dict(name="batch_padded", kind="padded", passes="both", irreps=WATER, lmax=3, out="0e+1o+2e+3o", system="water",
             atoms=192, neighbours=53, capacity=12288),
        # The 3000-atom water box of the benchmark, energy only.
        dict(name="water_fwd", kind="conv", passes="fwd", irreps=WATER, lmax=3, system="water", atoms=3000, neighbours=53.6),
        # The same box, the backward that forces need.
        dict(name="water_bwd", kind="conv", passes="bwd", irreps=WATER, lmax=3, system="water", atoms=3000, neighbours=53.6),
        # A large system of uneven density and an odd number of atoms, forward and backward.
        dict(name="large_skewed", kind="conv", passes="both", irreps=WATER, lmax=3, system="skewed", atoms=24001,
             neighbours=47),
        # High-order features: many coupling paths.
        dict(name="high_order", kind="conv", passes="both", irreps=HIGHORDER, lmax=3, system="liquid", atoms=1500,
             neighbours=52.2),
        # Streaming tensor product, an odd number of rows.
        dict(name="tensor_product", kind="tp", irreps=TP, lmax=3, rows=49157),
        # One step of training on forces: forward, backward, double backward.
        dict(name="force_training", kind="training", irreps=WATER, lmax=3, system="water", atoms=1029, neighbours=53),
        # The benchmark box from edge vectors and the radial network's hidden activations, forward and backward.
        dict(name="radial_layer", kind="radial", irreps=WATER, lmax=3, system="water", atoms=3000, neighbours=53.6, hidden=64),
        # A dynamics step of a smaller model on a middling box: new neighbour list, forward and backward.
        dict(name="md_step", kind="md", irreps="64x0e+64x1o", lmax=3, system="water", atoms=1536, neighbours=53),
        # A model whose signature has no kernels of its own: 48 channels, three input irreps, l <= 2.
        dict(name="own_signature", kind="conv", passes="both", irreps="48x0e+48x1o+48x2e", lmax=2, system="liquid", atoms=701,
             neighbours=50),
        # Double precision, as a geometry optimisation or a check of gradients uses it.
        dict(name="float64", kind="f64", irreps="64x0e+64x1o", lmax=2, system="water", atoms=192, neighbours=53),
    ]


# signatures with generated kernels: (irreps, lmax, output filter, collapsed outputs), and the largest graph drawn for each
_GENERATED = [
    (WATER, 3, "", False, 12000), (WATER, 3, "0e+1o+2e+3o", False, 12000), (WATER, 3, "", True, 8000),
    (WATER, 2, "", False, 12000), ("128x0e", 3, "", False, 16000), ("256x0e+256x1o", 3, "", False, 4000),
    ("96x0e+96x1o", 3, "", False, 6000), ("64x0e+64x1o", 3, "", False, 16000), ("32x0e+32x1o", 3, "", False, 16000),
    (HIGHORDER, 3, "", False, 2500), ("64x0e+64x1o+64x2e", 3, "", False, 4000), (TP, 3, "", False, 2000),
    ("128x0e+128x1o+128x2e+128x3o", 2, "", False, 2000),
]
_SOME_IRREPS = ["0e", "0e+1o", "0e+1o+2e", "0e+0o+1o+1e", "0e+1o+2e+3o"]


def _between(rng, lo, hi):
    """A whole number spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _graph_fields(rng, lo, hi):
    system = rng.choice(["water", "skewed", "liquid"])
    if system == "water":
        grid = max(4, int((_between(rng, lo, hi) / 3) ** (1 / 3)))
        atoms = 3 * grid ** 3
    else:
        atoms = _between(rng, lo, min(hi, 3000) if system == "liquid" else hi)
    return dict(system=system, atoms=atoms, neighbours=rng.randint(20, 47 if system == "skewed" else 53))


def _own_signature(rng, weights, lo):
    """A signature without generated kernels and a graph of at most `weights` edge weights."""
    while True:
        mul = 4 * rng.randint(1, 24)
        irreps, lmax = "+".join(f"{mul}x{ir}" for ir in rng.choice(_SOME_IRREPS).split("+")), rng.randint(1, 3)
        plan = _plan(dict(irreps=irreps, lmax=lmax))
        most = int(weights / (plan.n_paths * plan.n_channels * 53))
        if not plan.specialised and most > lo:
            return dict(irreps=irreps, lmax=lmax), min(most, 6000)


def draw(rng):
    """One more case: every kind, its sizes over the whole range, odd ones among them."""
    kind = rng.choice(["conv", "conv", "own", "padded", "md", "radial", "training", "tp", "f64"])
    if kind == "own":
        sig, most = _own_signature(rng, 6e7, 64)
        return dict(sig, kind="conv", passes=rng.choice(["fwd", "bwd", "both"]), **_graph_fields(rng, 64, most))
    if kind == "f64":
        if rng.random() < 0.5:
            sig, most = _own_signature(rng, 1.5e7, 64)
        else:
            sig, most = dict(irreps=rng.choice(["64x0e+64x1o", "32x0e+32x1o"]), lmax=rng.randint(1, 3)), 300
        return dict(sig, kind="f64", **_graph_fields(rng, 64, most))
    if kind == "tp":
        irreps, lmax, _, _, _ = rng.choice([s for s in _GENERATED if not s[3] and s[2] == ""])
        rows = _between(rng, 33, 49157)
        return dict(kind="tp", irreps=irreps, lmax=lmax, rows=rows if irreps == TP else min(rows, 32771))
    irreps, lmax, out, collapse, most = rng.choice(_GENERATED)
    if kind in ("radial", "training"):
        most //= 3
    sig = dict(irreps=irreps, lmax=lmax, out=out, collapse=collapse)
    case = dict(sig, kind=kind, **_graph_fields(rng, 64, most))
    if kind == "conv":
        case["passes"] = rng.choice(["fwd", "bwd", "both"])
    if kind == "padded":
        case["passes"] = rng.choice(["fwd", "both"])
        case["capacity"] = int(_edges(case) * rng.uniform(1.0, 1.3)) + rng.randint(0, 100)
    if kind == "radial":
        case["hidden"] = rng.choice([8, 20, 32, 64, 64, 64, 96, 128])
    return case


def _plan(case):
    out = case.get("out") or None
    flags = e3j.E3J_PLAN_COLLAPSE_OUTPUTS if case.get("collapse") else 0
    return e3j.e3j_plan_create(case["irreps"], case["lmax"], out, -1 if out else case["lmax"], flags)


def _edges(case):
    return int(case["atoms"] * case["neighbours"]) // 2 * 2


def _positions(case, seed):
    rng = np.random.Generator(np.random.PCG64([seed, 11]))
    n, system = case["atoms"], case["system"]
    if system == "water":       # molecules on a jittered lattice at the density of water
        return (*workloads.water_box(rng, round((n / 3) ** (1 / 3)), 3.104), 5.0)
    if system == "liquid":      # single atoms, 0.8 A apart at least
        box = max(24.64 * (n / 1500.0) ** (1 / 3), 10.5)
        return workloads.sort_by_cell(workloads.sequential_insertion(rng, n, box, 0.8), box, 4.0), box, 5.0
    if system == "skewed":      # a tenth of the molecules at twice the density
        box = max(105.0 * (n / 100_000.0) ** (1 / 3), 10.5)
        return workloads.sort_by_cell(workloads.skewed_water(rng, n, box), box, 5.0), box, 5.0
    box = 6.0 * (n / 64.0) ** (1 / 3)
    return rng.uniform(0, box, size=(n, 3)), box, 3.0


def _graph(case, seed):
    """senders, receivers (int32, sorted by receiver, then sender) and the edge vectors, on the GPU: the closest
    pairs in both directions."""
    pos, box, radius = _positions(case, seed)
    p, n_edges = torch.tensor(pos, device="cuda").remainder(box), _edges(case)
    snd, rcv, vec = [], [], []
    reach = radius * (max(1.0, case["neighbours"] / 45.0) ** (1 / 3) * 1.15 if case["system"] != "points" else 1.3)
    for lo in range(0, p.shape[0], 1024):
        v = p[lo:lo + 1024, None, :] - p[None, :, :]
        v -= box * torch.round(v / box)
        d2 = (v * v).sum(-1)
        i, j = torch.nonzero((d2 > 0) & (d2 < reach * reach), as_tuple=True)
        rcv.append(i + lo), snd.append(j), vec.append(v[i, j])
    snd, rcv, vec = torch.cat(snd), torch.cat(rcv), torch.cat(vec)
    d2 = (vec * vec).sum(-1)
    keep = torch.sort(torch.argsort(d2, stable=True)[:n_edges]).values   # a pair's two directions have one distance
    assert keep.numel() == n_edges, "the box holds fewer pairs than the case asks for"
    return snd[keep].int(), rcv[keep].int(), vec[keep].float().contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    plan, kind = _plan(case), case["kind"]
    real = torch.float64 if kind == "f64" else torch.float32
    randn = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=real)
    d, dp, P, D, nq = plan.d_in, plan.d_sh, plan.n_paths, plan.d_out, plan.n_channels
    state = dict(kind=kind, plan=plan, passes=case.get("passes", "both"))
    if kind == "tp":
        rows = case["rows"]
        state.update(x=randn(rows, d, nq), sh=randn(rows, dp), w=randn(rows, P, nq), g=randn(rows, D, nq))
        return state
    n = case["atoms"]
    senders, receivers, vec = _graph(case, seed)
    e = senders.numel()
    state.update(n=n, senders=senders, receivers=receivers, vec=vec, x=randn(n, d, nq), g=randn(n, D, nq))
    if kind not in ("md", "radial"):
        state["sh"] = e3j.e3j_harmonics_fwd(case["lmax"], vec).to(real)
    if kind == "radial":
        state["h"], state["W"] = randn(e, case["hidden"]), randn(case["hidden"], P * nq) / math.sqrt(case["hidden"])
    else:
        state["w"] = randn(e, P, nq)
    if kind == "training":
        state["ct"] = (randn(n, d, nq), randn(e, dp), randn(e, P, nq))
    if kind == "padded":
        pad = max(0, case["capacity"] - e)
        tail = lambda t, value: torch.cat([t, torch.full((pad, *t.shape[1:]), value, dtype=t.dtype, device=t.device)])
        state.update(senders=tail(senders, n), receivers=tail(receivers, n), sh=tail(state["sh"], 0), w=tail(state["w"], 0))
    if kind not in ("padded", "md"):
        state["graph"] = e3j.e3j_graph_prepare(n, senders, receivers)
    return state


def run(state):
    kind, plan, x, g = state["kind"], state["plan"], state["x"], state["g"]
    if kind == "tp":
        sh, w = state["sh"], state["w"]
        return e3j.e3j_tp_fwd(plan, x, sh, w), e3j.e3j_tp_bwd(plan, x, sh, w, g)
    edges = state["senders"], state["receivers"]
    if kind == "md":
        rowptr, perm, colptr = e3j.e3j_graph_prepare(state["n"], *edges)
        vec, w = state["vec"], state["w"]
        return (e3j.e3j_conv_vec_fwd(plan, x, vec, w, *edges, rowptr),
                e3j.e3j_conv_vec_bwd(plan, x, vec, w, *edges, g, rowptr, perm, colptr))
    if kind == "padded":
        rowptr, perm, colptr = e3j.e3j_graph_prepare_padded(state["n"], *edges)
        out = e3j.e3j_conv_fwd_padded(plan, x, state["sh"], state["w"], *edges, rowptr)
        if state["passes"] == "fwd":
            return out
        return out, e3j.e3j_conv_bwd_padded(plan, x, state["sh"], state["w"], *edges, g, rowptr, perm, colptr)
    rowptr, perm, colptr = state["graph"]
    if kind == "radial":
        args = plan, x, state["vec"], state["h"], state["W"], *edges
        return e3j.e3j_conv_radial_vec_fwd(*args, rowptr), e3j.e3j_conv_radial_vec_bwd(*args, g, rowptr, perm, colptr)
    args = plan, x, state["sh"], state["w"], *edges
    if kind == "f64":
        return e3j.e3j_conv_fwd_f64(*args, rowptr), e3j.e3j_conv_bwd_f64(*args, g, perm, colptr)
    out = e3j.e3j_conv_fwd(*args, rowptr) if state["passes"] != "bwd" else None
    grads = e3j.e3j_conv_bwd(*args, g, rowptr, perm, colptr) if state["passes"] != "fwd" else None
    if kind == "training":
        return out, grads, e3j.e3j_conv_bwd_bwd(*args, g, rowptr, perm, colptr, *state["ct"])
    return out, grads


def work(case):
    plan, kind = _plan(case), case["kind"]
    d, dp, P, D, nq = plan.d_in, plan.d_sh, plan.n_paths, plan.d_out, plan.n_channels
    size = 8 if kind == "f64" else 4
    n = case["rows"] if kind == "tp" else case["atoms"]
    e = case["rows"] if kind == "tp" else _edges(case)
    ids = 0 if kind == "tp" else 8 * e
    x, out = size * n * d * nq, size * n * D * nq
    angles = size * e * (3 if kind in ("md", "radial") else dp)
    weights = size * e * P * nq
    one = 2 * e * nq * (plan.n_pairs + D)        # a pass: every coefficient pair, every output row's edge scalar
    passes = case.get("passes", "both")
    flops = one * {"fwd": 1, "bwd": 3, "both": 4}[passes]
    if kind == "radial":                         # s = h W, and its two gradients
        hidden = case["hidden"]
        weights = size * (e * hidden + hidden * P * nq)
        flops += 3 * 2 * e * hidden * P * nq
    fwd = x + angles + weights + ids + out
    bwd = fwd + x + angles + weights
    total = (fwd if passes != "bwd" else 0) + (bwd if passes != "fwd" else 0)
    if kind in ("md", "padded"):                 # the list's pointers and the sender order
        total += 12 * e + 8 * n
    if kind == "padded" and passes != "fwd":     # zero gradients of the padding edges
        total += size * max(0, case["capacity"] - e) * (dp + P * nq)
    if kind == "training":                       # inputs and their cotangents in, four gradients out
        total += 3 * (x + angles + weights) + ids + 2 * out
        flops += 6 * one
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # About four times the largest errors of the calls against the float64 entry points on the same inputs: 3e-7 of the
    # norm and 4e-6 at one element in float32, 1.3e-6 and 5e-6 behind the radial layer's products (which carry 2^-22 of
    # every product); in float64 the same sums at that precision.
    if case["kind"] == "f64":
        return {"rel": 2e-15, "max": 3e-14}
    if case["kind"] == "radial":
        return {"rel": 5e-6, "max": 2e-5}
    return {"rel": 1.2e-6, "max": 1.6e-5}
