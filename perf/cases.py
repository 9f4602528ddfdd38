"""The work that a user of this library has it do, as cases that can be timed and compared.

A case names an entry point and its sizes.  References are SIFT-like descriptors laid out class by
class (or shuffled), as in ``paper_1112_0059_gb300/synth.py``, drawn on the GPU; the sizes are those
of the workloads there: the tiny set, the 101-class set (15 x 1,000 descriptors a class), the
256-class set (30 x 1,500 a class), and the query images of its batched and serving workloads.

``listed()``  the cases; ``draw(rng)`` one more of the same ranges; ``prepare(case, seed)`` the index,
the query descriptors and what else a program holds before the call; ``run(state)`` one call;
``work(case)`` the bytes and operations of a call; ``exact(case, seed)`` its outputs in 64 bits.
"""
from __future__ import annotations

import math

import torch

from paper_1112_0059_gb300 import lnbnn

DIM = 128
TINY = (10, 500)        # classes, descriptors a class
C101 = (101, 15000)
C256 = (256, 45000)


def _case(name, op, index, images, desc, k=10, shortlist=0, location_weight=-1, shuffled=False, workspace=False,
          beta=0.0, positive_only=False):
    """desc: (fewest, most) descriptors of an image."""
    case = {"op": op, "classes": index[0], "per_class": index[1], "images": images, "desc_lo": desc[0],
            "desc_hi": desc[1], "k": k, "shortlist": shortlist, "location_weight": location_weight,
            "shuffled": shuffled, "workspace": workspace, "beta": beta, "positive_only": positive_only}
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the tiny set: a call of a few thousand descriptors against a small index, where latency and launches count
        _case("tiny_batch", "local", TINY, 20, (100, 100)),
        # the smallest image of a server's stream, classified alone as it arrives: one query tile against every reference
        _case("lone_image", "local", C256, 1, (100, 100), workspace=True),
        # a server's median image alone, in its FP8 shortlist form
        _case("serve_fp8", "local", C256, 1, (632, 632), shortlist=24, workspace=True),
        # host arrays in, host arrays out: a few images of an application that keeps nothing on the GPU but the index
        _case("host_images", "host", C101, 5, (400, 1601)),
        # throughput on the largest index: a fifth of the benchmark's query set, exact
        _case("batch_exact", "local", C256, 100, (1500, 1500)),
        # the same index, images of uneven size in one call, FP8 shortlist
        _case("batch_fp8", "local", C256, 64, (200, 3000), shortlist=24),
        # a long shortlist (recall over speed), a server's batch of uneven images
        _case("fp8_m128", "local", C256, 10, (200, 3000), shortlist=128),
        # the paper's sweep over k: 50 neighbours, the 101-class set and its whole query set
        _case("k50_batch", "local", C101, 200, (1000, 1000), k=50),
        # the far end of that sweep: 100 neighbours, the 256-class set, a server's batch
        _case("k100_batch", "local", C256, 10, (1500, 1500), k=100),
        # original NBNN, the method compared against, on uneven images
        _case("nbnn_batch", "nbnn", C101, 20, (200, 1801)),
        # NBNN as a sum of log-odds increments, positive ones only (the paper's Table 1)
        _case("logodds", "logodds", C101, 8, (200, 1801), beta=1e-5, positive_only=True),
        # neighbours of location-weighted descriptors, an odd number of them, for a program's own scoring
        _case("located_knn", "knn", C101, 1, (3001, 3001), k=20, location_weight=10),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# pairs of query and reference descriptors of the largest listed case; long lists (which cost more a pair) and
# the log-odds rule (which writes a row of every class) stay below a share of it
_MOST_PAIRS = 100 * 1500 * 256 * 45000


def draw(rng):
    op = rng.choice(["local", "local", "local", "fp8", "fp8", "host", "nbnn", "logodds", "knn"])
    classes = _log_int(rng, 10, 256)
    per_class = _log_int(rng, 500, 45000)
    k = rng.choice([1, 2, 5, 10, 10, 20, 50, 100]) if op in ("local", "knn") else 10
    shortlist = rng.choice([24, 24, 32, 64, 128]) if op == "fp8" else 0
    located = rng.choice([-1, -1, 0, 10, 48]) if op in ("local", "knn", "nbnn") else -1
    longest = max(k + 1, shortlist)
    most = _MOST_PAIRS // (1 if longest <= 25 else 4 if longest <= 64 else 8)
    if op in ("host", "nbnn", "logodds"):
        most //= 8
    rows = _log_int(rng, 100, max(200, min(150000, most // (classes * per_class))))
    images = 1 if op == "knn" else _log_int(rng, 1, max(1, rows // 100))
    mean = max(1, rows // images)
    spread = rng.choice([0.0, 0.5, 0.85])
    return _case("", "local" if op == "fp8" else op, (classes, per_class), images,
                 (max(1, int(mean * (1 - spread))), max(1, int(mean * (1 + spread)))), k=k, shortlist=shortlist,
                 location_weight=located, shuffled=rng.random() < 0.25,
                 workspace=op in ("local", "fp8", "knn") and rng.random() < 0.4,
                 beta=rng.choice([1e-6, 1e-5, 1e-4]) if op == "logodds" else 0.0,
                 positive_only=op == "logodds" and rng.random() < 0.7)


def _counts(case):
    """Descriptors of each image, spread evenly over the case's range (the same for every seed)."""
    lo, hi = case["desc_lo"], case["desc_hi"]
    return [lo + int((hi - lo) * ((i * 0.6180339887498949 + 0.5) % 1.0) + 0.5) for i in range(case["images"])]


def _rows(proto, homes, cls, gen):
    """uint8 descriptors of the given classes: a prototype of the class, noise, zeroed coordinates."""
    n, dev = cls.shape[0], cls.device
    out = torch.empty((n, DIM + (2 if homes is not None else 0)), dtype=torch.uint8, device=dev)
    for at in range(0, n, 1 << 20):
        c = cls[at:at + (1 << 20)].long()
        pick = c * 16 + torch.randint(16, (c.shape[0],), generator=gen, device=dev)
        x = torch.randn((c.shape[0], DIM), generator=gen, device=dev).mul_(12.0).add_(proto[pick])
        x.mul_(torch.rand((c.shape[0], DIM), generator=gen, device=dev) >= 0.3)
        out[at:at + (1 << 20), :DIM] = x.clamp_(0, 255).round_().to(torch.uint8)
        if homes is not None:
            xy = torch.randn((c.shape[0], 2), generator=gen, device=dev).mul_(24.0).add_(homes[pick])
            out[at:at + (1 << 20), DIM:] = xy.clamp_(0, 255).round_().to(torch.uint8)
    return out


def _data(case, seed):
    """(references, labels, queries, offsets) on the GPU."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    C, n = case["classes"], case["classes"] * case["per_class"]
    pool = torch.rand((64, DIM), generator=gen, device=dev) * 128.0
    sel = torch.rand((C, 64), generator=gen, device=dev).argsort(dim=1)[:, :16].reshape(-1)
    proto = pool[sel] + 20.0 * torch.randn((C * 16, DIM), generator=gen, device=dev)
    located = case["location_weight"] >= 0
    homes = 32.0 + 192.0 * torch.rand((C * 16, 2), generator=gen, device=dev) if located else None
    labels = torch.arange(C, dtype=torch.int32, device=dev).repeat_interleave(case["per_class"])
    if case["shuffled"]:
        labels = labels[torch.randperm(n, generator=gen, device=dev)].contiguous()
    ref = _rows(proto, homes, labels, gen)
    counts = torch.tensor(_counts(case), dtype=torch.int64, device=dev)
    offsets = torch.zeros(len(counts) + 1, dtype=torch.int64, device=dev)
    offsets[1:] = counts.cumsum(0)
    img_cls = torch.randint(C, (len(counts),), generator=gen, device=dev, dtype=torch.int32)
    queries = _rows(proto, homes, img_cls.repeat_interleave(counts), gen)
    return ref, labels, queries, offsets


def prepare(case, seed):
    ref, labels, queries, offsets = _data(case, seed)
    located = case["location_weight"] >= 0
    index = lnbnn.Index(ref, labels, case["classes"], location_weight=case["location_weight"] if located else None)
    if case["shortlist"]:
        index.prepare_fp8()
    state = {"case": case, "index": index, "q": queries, "off": offsets, "ws": None, "out": None}
    m, n_img = queries.shape[0], case["images"]
    if case["op"] == "host":
        state["q"] = queries.cpu().pin_memory().numpy()
        state["off"] = offsets.cpu().pin_memory().numpy()
    elif case["workspace"]:
        # a server's slot: device scratch and result buffers kept from call to call
        state["ws"] = index.workspace(m, max(case["k"], case["shortlist"] - 1))
        shape = (m, case["k"]) if case["op"] == "knn" else (n_img, case["classes"])
        state["out"] = (torch.empty(shape, dtype=torch.int32 if case["op"] == "knn" else torch.int64, device="cuda"),
                        torch.empty(shape if case["op"] == "knn" else (n_img,), dtype=torch.int32, device="cuda"))
    return state


def run(state):
    case, index = state["case"], state["index"]
    op, q, off = case["op"], state["q"], state["off"]
    shortlist = case["shortlist"] or None
    if op == "local":
        return index.lnbnn_classify(q, off, case["k"], out=state["out"], workspace=state["ws"], shortlist=shortlist)
    if op == "knn":
        return index.knn_search(q, case["k"], out=state["out"], workspace=state["ws"])
    if op == "nbnn":
        return index.nbnn_classify(q, off)
    if op == "logodds":
        return index.nbnn_logodds_classify(q, off, case["beta"], positive_only=case["positive_only"])
    return index.classify_host(q, off, case["k"])


def work(case):
    """Every reference and query descriptor read once as its bytes, the results written once; the
    multiply-adds of the distance of every pair."""
    row = DIM + (2 if case["location_weight"] >= 0 else 0)
    n, m = case["classes"] * case["per_class"], sum(_counts(case))
    if case["op"] == "knn":
        results = 8 * m * case["k"]
    else:
        results = case["images"] * (8 * case["classes"] + 4 + (8 if case["op"] == "logodds" else 0))
        results += 8 * (case["images"] + 1)
    return {"bytes": row * (n + m) + results, "flops": 2 * row * n * m}


def _weighted(rows, weight):
    x = rows.double()
    if rows.shape[1] > DIM:
        x[:, DIM:] *= math.sqrt(weight)
    return x


def _sqdist(q, r):
    """Squared distances of whole numbers in 64 bits, rounded back to the whole numbers they are."""
    return ((q * q).sum(1)[:, None] + (r * r).sum(1)[None, :] - 2.0 * (q @ r.T)).round_()


def _neighbours(ref, queries, weight, k):
    """The k nearest as (row, distance), by distance and then by row."""
    best = torch.empty((queries.shape[0], 0), dtype=torch.int64, device=ref.device)
    q = _weighted(queries, weight)
    for at in range(0, ref.shape[0], 1 << 16):
        key = _sqdist(q, _weighted(ref[at:at + (1 << 16)], weight)).long() << 32
        key += torch.arange(at, at + key.shape[1], device=ref.device)
        best = torch.cat([best, key.topk(min(k, key.shape[1]), dim=1, largest=False).values], dim=1)
        best = best.topk(min(k, best.shape[1]), dim=1, largest=False).values
    best = best.sort(dim=1).values
    return best & 0xFFFFFFFF, best >> 32


def _class_minima(case, ref, labels, queries, weight):
    """[m, C] distance of the nearest reference of each class."""
    out = torch.full((queries.shape[0], case["classes"]), math.inf, dtype=torch.float64, device=ref.device)
    order = labels.argsort(stable=True)
    for c in range(case["classes"]):
        r = _weighted(ref[order[c * case["per_class"]:(c + 1) * case["per_class"]]], weight)
        for at in range(0, queries.shape[0], 4096):
            out[at:at + 4096, c] = _sqdist(_weighted(queries[at:at + 4096], weight), r).amin(dim=1)
    return out


def _per_image(rows, offsets):
    return torch.stack([rows[a:b].sum(0) for a, b in zip(offsets[:-1].tolist(), offsets[1:].tolist())])


def exact(case, seed):
    m, n = sum(_counts(case)), case["classes"] * case["per_class"]
    if case["shortlist"] or m * n > (3e10 if case["op"] in ("nbnn", "logodds") else 1e10):
        return None  # an approximate search (its results are whole numbers), or too long in 64 bits
    ref, labels, queries, offsets = _data(case, seed)
    weight, k = max(case["location_weight"], 0), case["k"]
    if case["op"] == "knn":
        idx, dist = _neighbours(ref, queries, weight, k)
        return idx.int(), dist.int()
    if case["op"] in ("local", "host"):
        idx, dist = _neighbours(ref, queries, weight, k + 1)
        lab, gain = labels[idx[:, :k]].long(), dist[:, :k] - dist[:, k:]
        seen = torch.zeros_like(gain, dtype=torch.bool)
        for b in range(1, k):
            seen[:, b] = (lab[:, :b] == lab[:, b:b + 1]).any(dim=1)
        rows = torch.zeros((m, case["classes"]), dtype=torch.int64, device=ref.device)
        rows.scatter_add_(1, lab, gain.masked_fill(seen, 0))
        totals = _per_image(rows, offsets)
        classes = totals.argmin(dim=1).int()
        return (totals.cpu(), classes.cpu()) if case["op"] == "host" else (totals, classes)
    d = _class_minima(case, ref, labels, queries, weight)
    if case["op"] == "nbnn":
        totals = _per_image(d.long(), offsets)
        return totals, totals.argmin(dim=1).int()
    # log P(C|d) P(Cbar) / P(Cbar|d) P(C) with the other classes summed for each class in turn
    x = -case["beta"] * d
    inc = torch.empty_like(x)
    for c in range(case["classes"]):
        others = torch.cat([x[:, :c], x[:, c + 1:]], dim=1)
        inc[:, c] = x[:, c] - torch.logsumexp(others, dim=1) + math.log(case["classes"] - 1)
    keep = inc > 0 if case["positive_only"] else torch.ones_like(inc, dtype=torch.bool)
    totals = _per_image(inc * keep, offsets)
    return totals, totals.argmax(dim=1).int(), _per_image(keep.long().sum(1), offsets)
