"""The work a user of this library has it do, as cases with sizes, inputs and one pass each.

Every pass goes through the Python package's public calls.  The kinds of work:

  analyse   the whole phenotype map of a box and what is read from it: designability, the Eq. 2
            numerators, the neutral networks and the Eq. 2 rows of two folds that are compared
  map       the phenotypes of a range of ids (a shard of a space too large for one map, a sample's
            neighbourhood, the training labels of the proposal), at any energy-gap threshold
  batch     several boxes' ranges captured once as a graph plan and replayed
  reduce    the reductions of a map that is already there (a shard of a streamed space)
  phi       the whole matrix of Eq. 2 numerators of such a map
  scan      the phenotypes of a list of ids: every conformation, or pruned by candidate classes
  propose   the proposal network's k best classes of a list of ids, and its logits
  train     one optimizer step of the proposal network, and the updated network's logits
"""
import functools
import math

import numpy as np
import torch

import paper_2008_05612_gb300 as hp
from paper_2008_05612_gb300 import inputs

BOXES = {"3x4": (3, 4), "2x2x3": (2, 2, 3), "4x4": (4, 4), "4x5": (4, 5), "5x5": (5, 5), "2x3x4": (2, 3, 4),
         "3x3x3": (3, 3, 3), "6x6": (6, 6)}
MAX_ROWS = 16384  # rows of the proposal network per step
PROBE = 64        # ids whose logits are read after an optimizer step


def listed():
    return [
        # the smallest whole job: a 16-residue box, where launches and read-backs are the time
        {"name": "analyse_4x4", "kind": "analyse", "box": "4x4"},
        # the paper's headline: all 2^27 sequences of 3x3x3 and every statistic of Section 3.2
        {"name": "analyse_3x3x3", "kind": "analyse", "box": "3x3x3"},
        # a ragged id range with the training labels (lowest minimiser) beside the phenotypes
        {"name": "map_ragged_3x3x3", "kind": "map", "box": "3x3x3", "count": 3_000_017, "aligned": False, "gap": 1,
         "aux": True},
        # one shard of the 6x6 space, as the shard streamer computes them
        {"name": "map_shard_6x6", "kind": "map", "box": "6x6", "count": 1 << 25, "aligned": True, "gap": 1, "aux": False},
        # a stability threshold above strict uniqueness, over a ragged range of 2x3x4
        {"name": "map_gap_2x3x4", "kind": "map", "box": "2x3x4", "count": 1_234_567, "aligned": False, "gap": 12,
         "aux": False},
        # small boxes together, replayed from a graph plan
        {"name": "batch_small", "kind": "batch", "boxes": "4x4,4x5,5x5", "bits": 25},
        # the reductions of a map at the 3x3x3 folding density
        {"name": "reduce_3x3x3", "kind": "reduce", "box": "3x3x3", "bits": 25},
        # the phenotype-to-phenotype matrix of such a map (0.9 million nonzero entries)
        {"name": "phi_3x3x3", "kind": "phi", "box": "3x3x3", "bits": 25},
        # the paper's sampling mode: random sequences against every conformation
        {"name": "scan_plain_3x3x3", "kind": "scan", "box": "3x3x3", "n": 16384, "k": 0, "gap": 1, "aux": True},
        # the same pruned by proposed classes, on the box where no exhaustive map applies
        {"name": "scan_pruned_6x6", "kind": "scan", "box": "6x6", "n": 65536, "k": 4, "gap": 1, "aux": False},
        # proposal inference, one full batch
        {"name": "propose_3x3x3", "kind": "propose", "box": "3x3x3", "width": 512, "n": 16384, "k": 4},
        # one optimizer step at the batch the proposal is trained with
        {"name": "train_3x3x3", "kind": "train", "box": "3x3x3", "width": 512, "n": 4096},
    ]


def _log(rng, lo, hi):
    """A whole number of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["analyse", "map", "map", "map", "batch", "reduce", "phi", "scan", "scan", "propose", "train"])
    if kind == "analyse":
        return {"kind": kind, "box": rng.choice(["4x4", "4x5", "5x5", "2x3x4"])}
    if kind == "map":
        box = rng.choice(["4x5", "5x5", "2x3x4", "3x3x3", "6x6"])
        top = min(1 << 24, (1 << math.prod(BOXES[box])) - 1)
        aligned = rng.random() < 0.4
        count = 1 << rng.randint(10, int(math.log2(top))) if aligned else _log(rng, 1, top // 4)
        return {"kind": kind, "box": box, "count": count, "aligned": aligned,
                "gap": rng.choice([1, 1, 1, rng.randint(2, 40)]), "aux": rng.random() < 0.4}
    if kind == "batch":
        boxes = rng.sample(["3x4", "2x2x3", "4x4", "4x5", "5x5", "2x3x4", "3x3x3"], rng.randint(2, 5))
        return {"kind": kind, "boxes": ",".join(boxes), "bits": rng.randint(12, 22)}
    if kind in ("reduce", "phi"):
        box = rng.choice(["5x5", "3x3x3", "6x6"])
        return {"kind": kind, "box": box, "bits": rng.randint(11, 25 if kind == "reduce" or box == "3x3x3" else 20)}
    if kind == "scan":
        box, k = rng.choice(["5x5", "3x3x3", "6x6"]), rng.choice([0, 1, 2, 4, 8])
        return {"kind": kind, "box": box, "n": _log(rng, 1, 65536 if k else 16384), "k": k,
                "gap": rng.choice([1, 1, rng.randint(2, 40)]), "aux": rng.random() < 0.5}
    case = {"kind": kind, "box": rng.choice(["5x5", "3x3x3", "6x6"]), "width": rng.choice([128, 256, 512])}
    if kind == "propose":
        return {**case, "n": _log(rng, 1, MAX_ROWS), "k": rng.randint(1, 16)}
    return {**case, "n": _log(rng, 32, 8192)}


# ---------------------------------------------------------------- what a program keeps or is given


@functools.lru_cache(maxsize=None)
def box_of(name):
    """The fold library of a box: enumerated once, as a program does, and used by every call."""
    return hp.Structs(BOXES[name])


def random_ids(N, n, seed):
    return torch.from_numpy(inputs.sample_ids(N, n, seed=seed).view(np.int64)).cuda()


@functools.lru_cache(maxsize=3)
def trained(box, width):
    """fp32 parameters of the proposal network after a short training in plain torch on uniform ids and
    their labels (lowest minimiser), so that logits and candidates look as they do in use."""
    s = box_of(box)
    batch, steps = 2048, 256
    ids = random_ids(s.N, batch * 16, 611)
    label = hp.sequence_scan(s, ids, aux=True)[1].long()
    x = ((ids[:, None] >> torch.arange(s.N, device="cuda")) & 1).float()
    shapes = [(width, s.N), (width,), (width, width), (width,), (s.S, width), (s.S,)]
    fan = [s.N, s.N, width, width, width, width]
    p = [torch.from_numpy(inputs.init_weights(sh, f, seed=71 + i)).float().cuda().requires_grad_()
         for i, (sh, f) in enumerate(zip(shapes, fan))]
    opt = torch.optim.Adam(p, lr=1e-3)
    for i in range(steps):
        b = slice((i % 16) * batch, (i % 16 + 1) * batch)
        h = torch.relu(torch.relu(x[b] @ p[0].T + p[1]) @ p[2].T + p[3])
        loss = torch.nn.functional.cross_entropy(h @ p[4].T + p[5], label[b])
        opt.zero_grad()
        loss.backward()
        opt.step()
    return [q.detach().cpu().numpy() for q in p]


def shard_map(box, bits, seed):
    """A map of 2^bits ids at the box's folding density: one aligned block of the space, with H and P
    swapped at residues chosen by the seed and the classes renumbered by the seed (a relabelling that
    keeps neighbours and networks, so that every seed's map has as many of them)."""
    s = box_of(box)
    rng = np.random.default_rng(seed)
    block = inputs.shard_index(0, 1 << (s.N - bits))
    flip = int(rng.integers(0, 1 << bits))
    phen = hp.phenotype_map(s, block << bits, 1 << bits)
    number = torch.from_numpy(np.append(rng.permutation(s.S), -1).astype(np.int32)).cuda()
    return number[phen[torch.arange(1 << bits, device="cuda") ^ flip].long()]


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    if kind == "batch":
        libs = [box_of(b) for b in case["boxes"].split(",")]
        ranges = []
        for s in libs:
            n = 1 << min(s.N, case["bits"])
            ranges.append((int(rng.integers(0, (1 << s.N) // n)) * n, n))
        # one ragged range among them, so that a plan holds several blocks of a box
        begin, n = ranges[-1]
        ranges[-1] = (begin + int(rng.integers(0, n // 5)), n - n // 5)
        outs = [torch.empty(n, dtype=torch.int32, device="cuda") for _, n in ranges]
        return {"kind": kind, "plan": hp.BatchPlan(libs, ranges, outs), "outs": outs}
    s = box_of(case["box"])
    if kind == "analyse":
        return {"kind": kind, "s": s, "q": rng.choice(s.S, 2, replace=False).tolist()}
    if kind == "map":
        count, space = case["count"], 1 << s.N
        begin = int(rng.integers(0, space // count)) * count if case["aligned"] else int(rng.integers(0, space - count + 1))
        return {"kind": kind, "s": s, "begin": begin, "count": count, "gap": case["gap"], "aux": case["aux"]}
    if kind in ("reduce", "phi"):
        return {"kind": kind, "s": s, "bits": case["bits"], "phen": shard_map(case["box"], case["bits"], seed)}
    ids = random_ids(s.N, case["n"], seed)
    if kind == "scan":
        cand = None
        if case["k"]:
            # proposals as a trained network makes them: the ground state of the sequence itself for
            # nine in ten, else (and in the other places) those of sequences one flip away
            bit = torch.from_numpy(rng.integers(0, s.N, (case["k"], case["n"]))).cuda()
            near = ids ^ (1 << bit)
            hit = torch.from_numpy(rng.random(case["n"]) < 0.9).cuda()
            near[0] = torch.where(hit, ids, near[0])
            top = hp.sequence_scan(s, near.reshape(-1), aux=True)[1].reshape(case["k"], -1).T.contiguous()
            cand = hp.proposal_conformations(s, top)
        return {"kind": kind, "s": s, "ids": ids, "cand": cand, "gap": case["gap"], "aux": case["aux"]}
    net = hp.MLP(s.N, case["width"], case["width"], s.S, MAX_ROWS if kind == "propose" else case["n"],
                 trained(case["box"], case["width"]))
    if kind == "propose":
        return {"kind": kind, "net": net, "ids": ids, "k": min(case["k"], s.S)}
    label = hp.sequence_scan(s, ids, aux=True)[1]
    return {"kind": kind, "net": net, "ids": ids, "label": label, "probe": ids[: min(PROBE, case["n"])].clone()}


# ---------------------------------------------------------------- one pass


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["plan"].launch()
        return state["outs"]
    if kind == "analyse":
        s = state["s"]
        phen = hp.phenotype_map(s)
        hist = hp.designability(phen, s.S)
        neutral, to_del = hp.robustness(phen, s.N, s.S)
        label, ncomp = hp.neutral_components(phen, s.N, s.S)
        rows = [hp.neighbourhood(phen, s.N, s.S, q) for q in state["q"]]
        return phen, hist, neutral, to_del, label, ncomp, *rows
    if kind == "map":
        out = [torch.empty(state["count"], dtype=torch.int32, device="cuda") for _ in range(2 if state["aux"] else 1)]
        hp.phenotype_map(state["s"], state["begin"], state["count"], out=out[0], aux=out[1] if state["aux"] else None,
                         gap_threshold=state["gap"])
        return out
    if kind == "reduce":
        phen, bits, S = state["phen"], state["bits"], state["s"].S
        hist = hp.designability(phen, S)
        neutral, to_del = hp.robustness(phen, bits, S)
        label, ncomp = hp.neutral_components(phen, bits, S)
        return hist, neutral, to_del, label, ncomp
    if kind == "phi":
        return hp.phi_matrix(state["phen"], state["bits"], state["s"].S)
    if kind == "scan":
        return hp.sequence_scan(state["s"], state["ids"], cand=state["cand"], aux=state["aux"], gap_threshold=state["gap"],
                                gaps=state["gap"] > 1)
    net = state["net"]
    if kind == "propose":
        return net.topk(state["ids"], state["k"]), net.logits(state["ids"][:PROBE])
    net.train_step(state["ids"], state["label"], 1e-3)
    return net.logits(state["probe"])


# ---------------------------------------------------------------- what a pass cannot do without


def library_bytes(s):
    return s.S_dir * (2 * s.C + 4)  # two residues per contact, a class per conformation


def work(case):
    """Inputs read once, outputs written once; a sequence's energy on its own ground state (C contacts,
    one multiply and one add each) for every phenotype that is computed."""
    kind = case["kind"]
    if kind == "batch":
        libs = [box_of(b) for b in case["boxes"].split(",")]
        ids = [1 << min(s.N, case["bits"]) for s in libs]
        return {"bytes": sum(4 * n + library_bytes(s) for s, n in zip(libs, ids)),
                "flops": sum(2 * s.C * n for s, n in zip(libs, ids))}
    s = box_of(case["box"])
    if kind == "analyse":
        n = 1 << s.N
        return {"bytes": library_bytes(s) + 4 * n + 4 * n + 8 * 6 * (s.S + 1), "flops": 2 * s.C * n}
    if kind == "map":
        return {"bytes": library_bytes(s) + 4 * case["count"] * (2 if case["aux"] else 1), "flops": 2 * s.C * case["count"]}
    if kind == "reduce":
        n = 1 << case["bits"]
        return {"bytes": 4 * n + 4 * n + 8 * 4 * (s.S + 1), "flops": case["bits"] * n}
    if kind == "phi":
        n = 1 << case["bits"]
        return {"bytes": 4 * n + 8 * (s.S + 2), "flops": case["bits"] * n}
    n = case["n"]
    if kind == "scan":
        outs = 1 + (1 if case["aux"] else 0) + (1 if case["gap"] > 1 else 0)
        return {"bytes": library_bytes(s) + n * (8 + 8 * case["k"] + 4 * outs), "flops": 2 * s.C * n}
    w = case["width"]
    params = w * s.N + w + w * w + w + s.S * w + s.S
    mul = w * s.N + w * w + s.S * w
    if kind == "propose":
        return {"bytes": 2 * params + n * (8 + 4 * case["k"]) + 4 * min(PROBE, n) * s.S, "flops": 2 * mul * (n + min(PROBE, n))}
    # forward, weight gradients and input gradients (none for the first layer's inputs); Adam reads and
    # writes the weights and both moments
    return {"bytes": 24 * params + 12 * n + 4 * min(PROBE, n) * s.S,
            "flops": 2 * (3 * mul - w * s.N) * n + 2 * mul * min(PROBE, n)}


def exact(case, seed):
    """The proposal's logits in 64 bits; nothing for whole-number outputs, and nothing after an optimizer
    step, whose first update is the sign of each gradient."""
    if case["kind"] != "propose":
        return None
    s = box_of(case["box"])
    ids = random_ids(s.N, case["n"], seed)[:PROBE]
    p = [torch.from_numpy(q).double().cuda() for q in trained(case["box"], case["width"])]
    x = ((ids[:, None] >> torch.arange(s.N, device="cuda")) & 1).double()
    h = torch.relu(torch.relu(x @ p[0].T + p[1]) @ p[2].T + p[3])
    return None, h @ p[4].T + p[5]
