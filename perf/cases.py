"""What a user has this library do, as timed cases.

Each case is one call (or one short sequence of calls) of the package's public
entry points on inputs of a size that the search, the exploratory search, the
learned proposal or the tests use:

  walk     a chunk of a search (search.run, the benchmark's step): walk every
           population, verify every best scheme on the device, collect each
           population's best scheme, read the counters and the rank histogram
  resize   one Resize move of the exploratory search (search.explore): a block
           of walkers transformed into another population's format
  window   window-mode steps (learned.evaluate), uniform or learned choice
  collect  the training data of the learned proposal (learned.collect)
  score    candidate rows scored by the proposal network
  grad     gradient and loss of the network on a batch of samples
  train    one optimiser step of the network (learned.train)

Walkers keep walking from pass to pass, as in a search; prepare() takes them
past the first steps from the start scheme, where nearly every flip is
accepted.  Walk results are integers and independent of how the work is laid
out on the GPU; the network's are floating point.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2511_20317_gb300 import learned, starts, tfg
from paper_2511_20317_gb300.workloads import MIXED_FORMATS, MIXED_RATIOS, largest_remainder_split, naive_start

PLATEAU = 50_000
STARTS = {"4x5x12": starts.start_4_5_12, "5x6x10": starts.start_5_6_10, "6x7x9": starts.start_6_7_9}


def listed():
    return [
        # the smallest search there is: (2,2,2), 1024 walkers, polled often
        {"name": "walk_222_1k", "kind": "walk", "pops": "2x2x2:0:1024", "steps": 1000, "burn": 500, "graph": 1,
         "policy": 0, "slack": 3},
        # the benchmark's step: (3,3,3) over Z_T and Z_2, 65536 walkers each, side by side
        {"name": "walk_333_131k", "kind": "walk", "pops": "3x3x3:0:65536,3x3x3:1:65536", "steps": 20000,
         "burn": 5000, "graph": 2, "policy": 0, "slack": 3},
        # five formats at once, the batched search
        {"name": "walk_mixed5_262k", "kind": "walk",
         "pops": ",".join("%dx%dx%d:0:%d" % (*f, n) for f, n in
                          zip(MIXED_FORMATS, largest_remainder_split(262144, MIXED_RATIOS))),
         "steps": 2000, "burn": 2000, "graph": 2, "policy": 0, "slack": 3},
        # large formats from meta-operator starts (terms of three words, ranks 202 to 351)
        {"name": "walk_large3_98k", "kind": "walk", "pops": "4x5x12:0:32768,5x6x10:0:32768,6x7x9:0:32768",
         "steps": 400, "burn": 800, "graph": 2, "policy": 0, "slack": 3},
        # the other walk policy (expansions after failed flips), both coefficient sets, ragged populations
        {"name": "walk_policy1_20k", "kind": "walk", "pops": "3x3x4:0:10007,2x4x5:1:9973", "steps": 2000,
         "burn": 1000, "graph": 1, "policy": 1, "slack": 6},
        # one Resize move on a whole population
        {"name": "resize_333_65k", "kind": "resize", "op": "extend", "src": "3x3x3", "axis": 2, "index": 0, "mode": 0,
         "walkers": 65536, "burn": 500},
        # uniform choice over the window (the comparator of the learned proposal)
        {"name": "window_444_262k", "kind": "window", "fmt": "4x4x4", "walkers": 262144, "steps": 20, "burn": 200,
         "policy": 0, "eps": 0.0},
        # learned choice over the window
        {"name": "learned_345_262k", "kind": "window", "fmt": "3x4x5", "walkers": 262144, "steps": 5, "burn": 200,
         "policy": 1, "eps": 0.05},
        # logged walks for training: small populations, many steps, a label horizon
        {"name": "collect_444_4k", "kind": "collect", "fmt": "4x4x4", "walkers": 4096, "steps": 500, "neg": 0.01,
         "horizon": 16},
        # the network on its own: scoring, gradient, one optimiser step at the training batch
        {"name": "score_1m", "kind": "score", "rows": 1_000_003},
        {"name": "grad_262k", "kind": "grad", "rows": 262_144},
        {"name": "train_8k", "kind": "train", "rows": 8192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


SMALL = ["2x2x2", "2x2x3", "2x3x3", "2x3x4", "3x3x3", "2x4x4", "2x4x5", "3x3x4", "3x4x5", "4x4x4", "4x4x5"]


def draw(rng):
    kind = rng.choice(["walk", "walk", "walk", "walk", "resize", "window", "window", "collect", "score", "grad",
                       "train"])
    if kind == "walk":
        policy = rng.choice([0, 0, 0, 1, 2])
        pops = []
        wide = rng.random() < 0.25
        for _ in range(rng.choice([1, 1, 2, 3])):
            fmt = rng.choice(sorted(STARTS) + ["4x5x5"]) if wide else rng.choice(SMALL)
            pops.append("%s:%d:%d" % (fmt, rng.choice([0, 0, 1]), _log_int(rng, 300, 16384 if wide else 50000)))
        return {"kind": kind, "pops": ",".join(pops), "steps": _log_int(rng, 50, 400 if wide else 2000),
                "burn": _log_int(rng, 50, 800), "graph": rng.choice([0, 1, 2]), "policy": policy,
                "slack": rng.choice([3, 4, 6])}
    if kind == "resize":
        return {"kind": kind, "op": rng.choice(["extend", "swap", "project", "double", "product", "merge"]),
                "src": rng.choice(["2x2x3", "2x3x3", "3x3x3", "2x3x4"]), "axis": rng.choice([0, 1, 2]),
                "index": rng.choice([1, 2, 3, 4, 5]), "mode": rng.choice([0, 0, 1]),
                "walkers": _log_int(rng, 300, 65536), "burn": _log_int(rng, 50, 800)}
    if kind == "window":
        policy = rng.choice([0, 1])
        return {"kind": kind, "fmt": rng.choice(SMALL), "walkers": _log_int(rng, 1000, 262144),
                "steps": _log_int(rng, 1, 5 if policy else 20), "burn": _log_int(rng, 20, 300), "policy": policy,
                "eps": 0.05 if policy else 0.0}
    if kind == "collect":
        return {"kind": kind, "fmt": rng.choice(SMALL), "walkers": _log_int(rng, 500, 8192),
                "steps": _log_int(rng, 50, 500), "neg": rng.choice([0.01, 0.05]), "horizon": rng.choice([1, 8, 16, 32])}
    return {"kind": kind, "rows": _log_int(rng, *{"score": (1, 4_000_000), "grad": (100, 500_000),
                                                  "train": (500, 65536)}[kind])}


# ---------------------------------------------------------------------------------------------
def _fmt(text):
    return tuple(int(x) for x in text.split("x"))


def _start(text, mode):
    s = STARTS[text]()[1] if text in STARTS else naive_start(*_fmt(text))
    return np.abs(s).astype(np.int8) if mode else s


def _state(W, pops=None):
    """Views of the walkers' device state, a population at a time: records, live
    slots, best slots (each padded to 256 bytes, the order of a checkpoint)."""
    used = ctypes.c_size_t()
    tfg._check(tfg.lib().tfg_checkpoint(W.ctx, None, 0, ctypes.byref(used)))
    off = W.workspace_bytes - used.value
    out = []
    for f, p in enumerate(W.pop):
        lt = tfg.term_len(p["fmt"])
        words = 1 if lt <= 64 else 3
        per = p["r_max"] * words * (4 if lt <= 32 else 8) * (1 if p["mode"] else 2)
        view = []
        for size in (p["walkers"] * tfg.WALKER_INFO_DTYPE.itemsize, p["walkers"] * per, p["walkers"] * per, per):
            view.append(W.workspace[off: off + size].view(torch.int32 if size % 8 else torch.int64))
            off += (size + 255) // 256 * 256
        if pops is None or f in pops:
            out.append({"records": view[0], "live": view[1], "best": view[2]})
    return out


def _params(**kw):
    return tfg.tfg_default_params(plateau_len=PLATEAU, **kw)


OPS = {"project": tfg.TFG_RESIZE_PROJECT, "extend": tfg.TFG_RESIZE_EXTEND, "double": tfg.TFG_RESIZE_DOUBLE,
       "merge": tfg.TFG_RESIZE_MERGE, "product": tfg.TFG_RESIZE_PRODUCT, "swap": tfg.TFG_RESIZE_SWAP}
ORDERS = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]


def _resize_target(case, src):
    """(result format, aux scheme, index) of a Resize move on format src."""
    op, a = case["op"], case["axis"]
    if op == "swap":
        return tuple(src[b] for b in ORDERS[case["index"]]), None, case["index"]
    if op == "project":
        return tuple(src[b] - (b == a) for b in range(3)), None, case["index"] % src[a]
    if op == "extend":
        return tuple(src[b] + (b == a) for b in range(3)), None, 0
    if op == "double":
        return tuple(src[b] * (2 if b == a else 1) for b in range(3)), None, 0
    if op == "merge":
        return (tuple(src[b] * (2 if b == a else 1) for b in range(3)),
                (src, _start("%dx%dx%d" % src, case["mode"])), 0)
    aux = (1, 1, 2)
    return tuple(src[b] * aux[b] for b in range(3)), (aux, naive_start(*aux)), 0


def _samples(case, seed):
    """Feature rows as the walks log them: counts, one-hot and flag columns, and
    the format's sizes; labels of a rare event and class-balanced weights."""
    g = np.random.default_rng([seed, case["rows"]])
    n = case["rows"]
    x = np.zeros((n, 32), np.float32)
    x[np.arange(n), g.integers(0, 3, n)] = 1.0
    x[:, 3:5] = g.integers(0, 2, (n, 2))
    x[:, 5:16] = g.integers(0, 9, (n, 11))
    x[:, 16:18] = g.random((n, 2)) < 0.02
    x[:, 18] = g.integers(2, 20, n)
    x[:, 19:24] = (2, 60, 4, 4, 4)
    x[:, 19] = g.integers(0, 3, n)
    x[:, 20] = g.integers(50, 65, n)
    x[:, 24] = g.integers(0, 65, n)
    x[:, 31] = 1.0
    lab = (g.random(n) < 0.1).astype(np.float32)
    pos = max(lab.sum(), 1.0)
    wt = np.where(lab > 0, 0.5 / pos, 0.5 / max(n - lab.sum(), 1.0)).astype(np.float32)
    return x, lab, wt


def _network(seed):
    """A parameter blob with every part non-zero (device bytes)."""
    blob = learned.init_params(seed).cpu().numpy()
    g = np.random.default_rng([seed, 77])
    vec = blob[40960: 40960 + 385 * 4].view(np.float32)
    vec[:256] = g.normal(0, 0.1, 256)
    vec[384] = 0.1
    return torch.from_numpy(blob).cuda()


def _split(blob):
    """The blob's parts: W1, W2 (bf16), then b1, b2, w3, b3 (float32)."""
    w = blob[:40960].view(torch.bfloat16)
    return {"W1": w[:4096].view(32, 128), "W2": w[4096:].view(128, 128),
            "vectors": blob[40960: 40960 + 385 * 4].view(torch.float32)}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "walk":
        pops = []
        for text in case["pops"].split(","):
            fmt, mode, n = text.split(":")
            pops.append((_fmt(fmt), int(mode), _start(fmt, int(mode)), int(n)))
        W = tfg.Walkers(pops, seed=seed, params=_params(use_graph=case["graph"], walk_policy=case["policy"],
                                                        expand_thresh=int(0.01 * 2**32) if case["policy"] == 1 else 0,
                                                        r_slack=case["slack"]))
        W.walk(case["burn"]).sync()
        return {"case": case, "W": W, "state": _state(W)}
    if kind == "resize":
        src = _fmt(case["src"])
        dst, aux, index = _resize_target(case, src)
        n = case["walkers"]
        pops = [(f, case["mode"], _start("%dx%dx%d" % f, case["mode"]), n) for f in (src, dst)]
        W = tfg.Walkers(pops, seed=seed, params=_params(r_slack=8))
        W.walk(case["burn"]).sync()
        return {"case": case, "W": W, "aux": aux, "index": index, "state": _state(W, (1,))}
    if kind == "window":
        fmt = _fmt(case["fmt"])
        W = tfg.Walkers([(fmt, 0, naive_start(*fmt), case["walkers"])], seed=seed, params=_params())
        W.walk(case["burn"]).sync()
        return {"case": case, "W": W, "net": _network(seed) if case["policy"] else None, "state": _state(W)}
    if kind == "collect":
        return {"case": case, "seed": seed}
    x, lab, wt = (torch.from_numpy(a).cuda() for a in _samples(case, seed))
    s = {"case": case, "net": _network(seed), "x": x.bfloat16(), "label": lab, "weight": wt}
    if kind == "train":
        s["trainer"] = tfg.MlpTrainer(s["net"])
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "walk":
        W = state["W"]
        W.walk(case["steps"])
        fails = W.verify_all()
        best = [W.collect_best(f) for f in range(W.n_formats)]
        counts, hist = W.stats()
        return {"state": state["state"], "fails": fails, "best": best, "counts": list(counts.values()), "hist": hist}
    if kind == "resize":
        W = state["W"]
        skipped = W.resize(OPS[case["op"]], 0, W.pop[1]["first"], case["walkers"], axis=case["axis"],
                           index=state["index"], aux=state["aux"], use_best=True)
        return {"state": state["state"], "skipped": skipped}
    if kind == "window":
        W = state["W"]
        chosen = W.walk_window(case["steps"], policy=case["policy"], mlp_params=state["net"],
                               eps_thresh=int(case["eps"] * 2**32), record_choices=True)
        W.sync()
        return {"state": state["state"], "chosen": chosen}
    if kind == "collect":
        e = learned.collect(formats=[_fmt(case["fmt"])], walkers=case["walkers"], steps=case["steps"],
                            seed=state["seed"], neg_rate=case["neg"], horizon=case["horizon"])
        # as many entries as are kept differs from seed to seed: the table ends in empty ones
        table = np.zeros(int(case["walkers"] * case["steps"] * (2 * case["neg"] + 0.02)) + 2000, e.dtype)
        table[:len(e)] = e
        return {"count": len(e), "feat": table["feat"], "label": table["label"], "walker": table["walker_id"],
                "step": table["step"]}
    if kind == "score":
        return tfg.tfg_mlp_score(state["net"], state["x"])
    if kind == "grad":
        grad, loss = tfg.tfg_mlp_grad(state["net"], state["x"], state["label"], state["weight"])
        return {"grad": grad, "loss": loss}
    tr = state["trainer"]
    tr.step(state["x"], state["label"], state["weight"], 2e-3)
    return {**_split(state["net"]), "loss": tr.state[4 * tfg.MLP_NUM_PARAMS: 4 * tfg.MLP_NUM_PARAMS + 1]}


def work(case):
    """Bytes read and written once, and the products' operations.  A walk reads
    and writes its walkers' records and live schemes; its steps are integer work
    on chip, which neither number counts."""
    kind = case["kind"]
    if kind in ("walk", "resize", "window", "collect"):
        if kind == "walk":
            pops = [(_fmt(t.split(":")[0]), int(t.split(":")[1]), int(t.split(":")[2])) for t in case["pops"].split(",")]
        else:
            f = _fmt(case["src" if kind == "resize" else "fmt"])
            pops = [(f, case.get("mode", 0), case["walkers"])]
        total = 0.0
        for (m, n, p), mode, walkers in pops:
            lt = m * n + n * p + p * m
            term = (4 if lt <= 32 else 8 * (1 if lt <= 64 else 3)) * (1 if mode else 2)
            total += walkers * 2.0 * (tfg.WALKER_INFO_DTYPE.itemsize + m * n * p * term)
        flops = 0.0
        if kind == "window" and case["policy"]:
            # the window's rows: the candidates of the terms, at most 256 (about 3 a term in a long walk)
            rows = min(256, 3 * _fmt(case["fmt"])[0] * _fmt(case["fmt"])[1] * _fmt(case["fmt"])[2])
            flops = case["steps"] * case["walkers"] * rows * 2.0 * (32 * 128 + 128 * 128 + 128)
        return {"bytes": total, "flops": flops}
    n = case["rows"]
    forward, backward = n * 2.0 * (32 * 128 + 128 * 128 + 128), n * 2.0 * (2 * 128 * 128 + 32 * 128 + 128)
    if kind == "score":
        return {"bytes": n * 68.0 + 42512, "flops": forward}
    out = 4.0 * 20866 if kind == "grad" else 42512 + 6 * 4.0 * 20865
    return {"bytes": n * 72.0 + 42512 + out, "flops": forward + backward}


def exact(case, seed):
    """The network's results in 64 bits (walk results are integers)."""
    if case["kind"] not in ("score", "grad", "train"):
        return None
    x, lab, wt = _samples(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x, lab, wt = (torch.from_numpy(a).to(dev).double() for a in (x, lab, wt))
    parts = _split(_network(seed).to(dev))
    W1, W2, vec = (parts[k].double().requires_grad_() for k in ("W1", "W2", "vectors"))

    def score(rows):
        h = torch.relu(rows @ W1 + vec[:128])
        h = torch.relu(h @ W2 + vec[128:256])
        return h @ vec[256:384] + vec[384]

    if case["kind"] == "score":
        with torch.no_grad():
            return torch.cat([score(rows) for rows in x.split(1 << 18)])
    loss = 0.0
    for a in range(0, x.shape[0], 1 << 17):
        sl = slice(a, a + (1 << 17))
        part = (wt[sl] * torch.nn.functional.softplus(-(2 * lab[sl] - 1) * score(x[sl]))).sum()
        part.backward()
        loss += float(part.detach())
    grads = [W1.grad, W2.grad, vec.grad]
    if case["kind"] == "grad":
        return {"grad": torch.cat([v.reshape(-1) for v in grads]), "loss": loss}
    new = [w.detach() - 2e-3 * g / (g.abs() + 1e-8) for w, g in zip((W1, W2, vec), grads)]
    return {"W1": new[0], "W2": new[1], "vectors": new[2], "loss": loss}
