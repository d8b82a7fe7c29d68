"""What a planner has this library do, as cases that can be timed.

A case is one unit of work of such a program, taken through the public entry points of
``paper_2510_18546_b200.enl``: a planning step, a scoring pass, a few decoded tokens, an update of the map, a step
with the slow tier, a tick that may not allocate.  Shapes (group lengths, select lists, rows per episode) follow from the case
alone, values from the seed alone.  Scores have a standard deviation of about 1.5 before the softmax, as attention
logits have, so that rows have a few dominant keys and running maxima move; in the scoring cases three objects of
four belong to a group and the rest to none.
"""
import functools
import math

import numpy as np
import torch

from paper_2510_18546_b200 import enl

BF16 = torch.bfloat16
MODEL = dict(q_heads=32, kv_heads=8, head_dim=128)            # the planner model of the benchmark configurations
OBJECT_TOKENS = 32                                            # tokens of a newly detected object's description
SCORE_STD = 1.5


def listed():
    return [
        # the smallest call: one layer of a small model, four short groups and a short instruction
        dict(MODEL, name="tiny_step", kind="plan", layers=1, q_heads=8, kv_heads=2, head_dim=64, shapes=10, batch=1, pool=16,
             sel=4, len_lo=32, len_hi=32, q_lo=64, q_hi=64, prior=0, mass=True),
        # an ordinary planning step: the selected part of the map, instruction and trajectory, every layer of the model
        dict(MODEL, name="planner_step", kind="plan", layers=40, shapes=11, batch=1, pool=200, sel=24, len_lo=40, len_hi=120,
             q_lo=512, q_hi=512, prior=0, mass=True),
        # a long episode: three times the map, twice the trajectory
        dict(MODEL, name="long_step", kind="plan", layers=40, shapes=12, batch=1, pool=128, sel=64, len_lo=20, len_hi=200,
             q_lo=1024, q_hi=1024, prior=0, mass=True),
        # sixteen robots planned for at once, prompts of different lengths
        dict(MODEL, name="concurrent_step", kind="plan", layers=10, shapes=13, batch=16, pool=40, sel=32, len_lo=40, len_hi=160,
             q_lo=256, q_hi=768, prior=0, mass=True),
        # clustering: new objects against every group of a large map on a tenth of the layers, masses kept per layer
        dict(MODEL, name="scoring_pass", kind="score", layers=4, shapes=14, groups=1000, len_lo=20, len_hi=200, n_q=1024,
             sums=False),
        # the same on an ordinary map where only the objects' averages are wanted: no outputs, sums taken on the way
        dict(MODEL, name="scoring_sums", kind="score", layers=4, shapes=15, groups=200, len_lo=40, len_hi=120, n_q=512,
             sums=True),
        # the plan is written token by token: after an ordinary step ...
        dict(MODEL, name="decode_short", kind="decode", layers=40, shapes=16, batch=1, pool=40, sel=24, len_lo=40, len_hi=120,
             new_lo=530, new_hi=530, tokens=3, mass=False),
        # ... over a large part of the map ...
        dict(MODEL, name="decode_long", kind="decode", layers=40, shapes=17, batch=1, pool=104, sel=96, len_lo=256, len_hi=426,
             new_lo=64, new_hi=64, tokens=2, mass=True),
        # ... and for sixteen robots at once
        dict(MODEL, name="decode_batch", kind="decode", layers=20, shapes=18, batch=16, pool=36, sel=32, len_lo=40, len_hi=160,
             new_lo=1, new_hi=128, tokens=2, mass=True),
        # the map changes: groups are rewritten and new objects join them (rotated, attended to the group, appended)
        dict(MODEL, name="map_update", kind="update", layers=20, shapes=19, groups=24, touched=4, len_lo=40, len_hi=120,
             add_lo=17, add_hi=61, per_layer=False),
        # the map does not fit: retrieval picks groups under a budget, the missing ones come from host memory
        dict(MODEL, name="tier_step", kind="tier", layers=20, shapes=20, groups=64, len_lo=40, len_hi=120, share=0.35, n_q=128),
        # a control loop that may not allocate: one token over contiguous keys, layer by layer
        dict(MODEL, name="static_tick", kind="static", layers=20, shapes=21, segs=24, len_lo=40, len_hi=120, new=530, mass=True),
    ]


# ---- more cases of the same ranges ------------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    heads = rng.choice([(32, 8, 128)] * 4 + [(8, 2, 64), (16, 2, 128), (8, 8, 64)])
    case = dict(q_heads=heads[0], kv_heads=heads[1], head_dim=heads[2], shapes=rng.randrange(1 << 20))
    lo = _log(rng, 8, 120)
    hi = int(lo * rng.uniform(1.2, 4.0)) + 1
    kind = rng.choice(["plan"] * 6 + ["score"] * 3 + ["decode"] * 6 + ["update"] * 2 + ["tier"] + ["static"] * 2)
    if kind == "plan":
        batch = 1 if rng.random() < 0.7 else rng.randint(2, 16)
        q_hi = _log(rng, 16, 1024)
        sel = _log(rng, 2, 96)
        case.update(kind=kind, layers=_log(rng, 1, 40), batch=batch, pool=sel + _log(rng, 1, 32), sel=sel, len_lo=lo, len_hi=hi,
                    q_lo=q_hi if batch == 1 else max(1, q_hi // 3), q_hi=q_hi, prior=0 if rng.random() < 0.7 else _log(rng, 1, 512),
                    mass=rng.random() < 0.7)
    elif kind == "score":
        case.update(kind=kind, layers=rng.randint(1, 4), groups=_log(rng, 64, 1000), len_lo=max(lo, 20), len_hi=min(max(hi, 40), 200),
                    n_q=_log(rng, 48, 1024), sums=rng.random() < 0.5)
        case["len_lo"] = min(case["len_lo"], case["len_hi"])
    elif kind == "decode":
        sel = _log(rng, 4, 128)
        new_hi = _log(rng, 1, 700)
        batch = 1 if rng.random() < 0.5 else rng.randint(2, 32)
        case.update(kind=kind, layers=_log(rng, 8, 40), batch=batch, pool=sel + rng.randint(0, 8), sel=sel, len_lo=lo, len_hi=hi,
                    new_lo=max(1, new_hi // 4) if batch > 1 else new_hi, new_hi=new_hi, tokens=rng.randint(2, 4), mass=rng.random() < 0.5)
    elif kind == "update":
        add = _log(rng, 8, 96)
        groups = _log(rng, 6, 64)
        case.update(kind=kind, layers=_log(rng, 4, 40), groups=groups, touched=rng.randint(1, 4), len_lo=lo, len_hi=hi,
                    add_lo=max(1, add // 2), add_hi=add, per_layer=rng.random() < 0.25)
    elif kind == "tier":
        case.update(kind=kind, layers=_log(rng, 4, 24), groups=_log(rng, 24, 96), len_lo=max(lo, 16), len_hi=max(hi, 20),
                    share=round(rng.uniform(0.2, 0.5), 2), n_q=_log(rng, 32, 256))
        case["len_hi"] = min(case["len_hi"], 160)
        case["len_lo"] = min(case["len_lo"], case["len_hi"])
    else:
        case.update(kind=kind, layers=_log(rng, 4, 40), segs=_log(rng, 1, 128), len_lo=lo, len_hi=hi, new=_log(rng, 1, 700),
                    mass=rng.random() < 0.7)
    # no dearer than the largest listed case, and small enough to hold three times
    while case["layers"] > 1 and (work(case)["flops"] > 4e12 or work(case)["bytes"] > 8e9 or _pool_bytes(case) > 1.0e10 or
                                  (kind == "tier" and _pool_bytes(case) > 6e8)):
        case["layers"] = max(1, case["layers"] * 3 // 4)
    while kind == "plan" and work(case)["flops"] > 4e12:
        case["q_lo"], case["q_hi"] = max(1, case["q_lo"] // 2), max(1, case["q_hi"] // 2)
    return case


# ---- shapes -----------------------------------------------------------------------------------------------------
def _lens(rng, n, case):
    return rng.integers(case["len_lo"], case["len_hi"] + 1, n).astype(np.int64)


def _shapes(case):
    """Group lengths, select lists and rows per episode, from the case's own `shapes` number."""
    return _shapes_of(tuple(sorted((k, v) for k, v in case.items() if k != "name")))


@functools.lru_cache(maxsize=64)
def _shapes_of(items):
    case = dict(items)
    rng = np.random.default_rng(case["shapes"])
    kind = case["kind"]
    if kind in ("plan", "decode"):
        b = case["batch"]
        lens = [_lens(rng, case["pool"], case) for _ in range(b)]
        sel = [rng.permutation(case["pool"])[:case["sel"]] for _ in range(b)]
        if kind == "plan":
            rows = [int(x) for x in rng.integers(case["q_lo"], case["q_hi"] + 1, b)]
            return dict(lens=lens, sel=sel, n_q=rows, n_new=[r + case["prior"] for r in rows])
        return dict(lens=lens, sel=sel, n_new=[int(x) for x in rng.integers(case["new_lo"], case["new_hi"] + 1, b)])
    if kind == "score":
        n_obj = -(-case["n_q"] // OBJECT_TOKENS)
        target = rng.integers(0, case["groups"], n_obj)
        target[rng.random(n_obj) < 0.25] = -1                  # these open a new group
        off = [min(i * OBJECT_TOKENS, case["n_q"]) for i in range(n_obj + 1)]
        return dict(lens=[_lens(rng, case["groups"], case)], sel=[np.arange(case["groups"])], n_q=[case["n_q"]],
                    n_new=[case["n_q"]], target=target, obj_off=off)
    if kind == "update":
        touched = rng.permutation(case["groups"])[:min(case["touched"], case["groups"])]
        return dict(lens=[_lens(rng, case["groups"], case)], touched=[int(g) for g in touched],
                    add=[int(x) for x in rng.integers(case["add_lo"], case["add_hi"] + 1, len(touched))])
    if kind == "tier":
        lens = _lens(rng, case["groups"], case)
        p0 = rng.random(case["groups"]).astype(np.float32)
        p1 = (0.5 * p0 + 0.5 * rng.random(case["groups"])).astype(np.float32)       # the robot has moved on a little
        mem = lens * _token_bytes(case) * case["layers"]
        budget = int(mem.sum() * case["share"])
        quantum = max(1 << 16, budget // 1024)
        chosen = [_knapsack(p, 0.2, mem, budget, quantum) for p in (p0, p1)]
        return dict(lens=[lens], prob=(p0, p1), threshold=0.2, mem=mem, budget=budget, quantum=quantum, chosen=chosen)
    return dict(seg_len=_lens(rng, case["segs"], case))


def _knapsack(prob, threshold, mem, budget, quantum):
    """The retrieval's choice, for the work figures only."""
    cap = budget // quantum
    best = np.zeros(cap + 1)
    take = np.zeros((len(prob), cap + 1), bool)
    for i, (p, m) in enumerate(zip(prob, mem)):
        v, w = float(p) - threshold, int(-(-int(m) // quantum))
        if v <= 0 or w > cap:
            continue
        with_i = np.concatenate([np.full(w, -1.0), best[:cap + 1 - w] + v])
        take[i] = with_i > best
        best = np.maximum(best, with_i)
    out, c = [], cap
    for i in range(len(prob) - 1, -1, -1):
        if take[i, c]:
            out.append(i)
            c -= int(-(-int(mem[i]) // quantum))
    return out[::-1]


def _token_bytes(case):
    return 4 * case["kv_heads"] * case["head_dim"]             # K and V of one token in one layer


def _pool_bytes(case):
    s = _shapes(case)
    n = int(sum(x.sum() for x in s["lens"])) if "lens" in s else int(s["seg_len"].sum()) + case["new"]
    return n * _token_bytes(case) * case["layers"]


# ---- what a pass cannot do without --------------------------------------------------------------------------------
def _attend_work(case, cached, n_q, n_new, slots, mass, out=True):
    hq, d = case["q_heads"], case["head_dim"]
    pairs = n_q * cached + n_q * (n_new - n_q) + n_q * (n_q + 1) / 2
    flops = (4.0 if out else 2.0) * hq * d * pairs
    rows = 2.0 * n_q * hq * d * (2 if out else 1)
    return np.array([(cached + n_new) * _token_bytes(case) + rows + (4.0 * n_q * hq * slots if mass else 0.0), flops])


def work(case):
    s, layers, kind = _shapes(case), case["layers"], case["kind"]
    w = np.zeros(2)
    if kind == "plan":
        for b in range(case["batch"]):
            w += layers * _attend_work(case, s["lens"][b][s["sel"][b]].sum(), s["n_q"][b], s["n_new"][b], case["sel"] + 1, case["mass"])
        w[0] += 2.0 * layers * _token_bytes(case) * s["lens"][0][s["sel"][0][0]]            # the group that is rewritten
    elif kind == "score":
        g = case["groups"]
        w += layers * _attend_work(case, s["lens"][0].sum(), case["n_q"], case["n_q"], g + 1, not case["sums"], out=not case["sums"])
        w[0] += 2.0 * layers * _token_bytes(case) * s["lens"][0][0] + 4.0 * (len(s["obj_off"]) - 1) * (g + 1)
        if case["sums"]:
            w[0] += 4.0 * case["n_q"] * case["q_heads"] * (g + 1)                          # one mass buffer for all layers
    elif kind == "decode":
        for b in range(case["batch"]):
            for j in range(case["tokens"]):
                w += layers * _attend_work(case, s["lens"][b][s["sel"][b]].sum(), 1, s["n_new"][b] + j, case["sel"] + 1, case["mass"])
    elif kind == "update":
        total = int(s["lens"][0].sum())
        for g, n in zip(s["touched"], s["add"]):
            have = int(s["lens"][0][g])
            total += n
            w += layers * _attend_work(case, have, n, n, 2, False)
            w[0] += layers * (2.0 * _token_bytes(case) * (have + n) + 4.0 * n * (case["q_heads"] + case["kv_heads"]) * case["head_dim"])
        w += layers * _attend_work(case, total, 1, 1, len(s["lens"][0]) + 1, False)
    elif kind == "tier":
        for k in (0, 1):
            sel = s["chosen"][k]
            w += layers * _attend_work(case, s["lens"][0][sel].sum(), case["n_q"], case["n_q"], len(sel) + 1, False)
            missing = [g for g in sel if g not in s["chosen"][1 - k]]
            w[0] += 2.0 * layers * _token_bytes(case) * s["lens"][0][missing].sum()
    else:
        w += layers * _attend_work(case, s["seg_len"].sum(), 1, case["new"], case["segs"] + 1, case["mass"])
    return {"bytes": float(w[0]), "flops": float(w[1])}


def tolerance(case):
    if case["kind"] == "score" and case["sums"]:
        return {"rel": 3e-5}                                    # fp32 masses of fp32 scores, and their averages
    return {"rel": 1e-2}                                        # bf16 outputs


# ---- inputs -------------------------------------------------------------------------------------------------------
class State:
    """A cache filled with the map, and the tensors of one pass."""

    def __init__(self, case):
        self.case, self.cache = case, None

    def __del__(self):
        if self.cache:
            enl.enl_cache_free(self.cache)
            self.cache = None


def _randn(gen, shape, sigma=1.0):
    x = torch.randn(shape, generator=gen, device="cuda", dtype=BF16)
    return x.mul_(sigma) if sigma != 1.0 else x


def _rows(gen, layers, n, heads, d, sigma=1.0):
    return _randn(gen, (layers, n, heads, d), sigma)


def _per_layer(x):
    return list(x.unbind(0))


def _queries(gen, case, n):
    return _rows(gen, case["layers"], n, case["q_heads"], case["head_dim"], SCORE_STD)


def _fill(case, state, gen, lens, max_batch, max_q, extra=0, capacity=None, affinity=None, evict=False):
    """Creates the cache and stores every group; returns the rows of the groups in `state.keep`, per layer."""
    layers, hkv, d = case["layers"], case["kv_heads"], case["head_dim"]
    lens = np.concatenate(lens)
    state.cache = enl.enl_cache_create(layers, case["q_heads"], hkv, d, len(lens), capacity or int(lens.sum()) + extra,
                                       device=torch.cuda.current_device(), max_batch=max_batch, max_q_tokens=max(max_q, 1))
    if evict:
        enl.enl_tier_enable(state.cache, int(lens.sum()))
    stream = torch.cuda.current_stream().cuda_stream
    rows = {}
    chunk = max(1, int(2e9 // max(1, layers * _token_bytes(case) * int(lens.max()))))
    for first in range(0, len(lens), chunk):
        part = lens[first:first + chunk]
        k = _rows(gen, layers, int(part.sum()), hkv, d)
        v = _rows(gen, layers, int(part.sum()), hkv, d)
        if affinity is not None:                                # keys of a group share a direction
            index = torch.repeat_interleave(torch.arange(len(part)), torch.from_numpy(part)).cuda()
            k += affinity[first:first + len(part)][index]
        kl, vl = _per_layer(k), _per_layer(v)
        at = 0
        for i, n in enumerate(part):
            n = int(n)
            ks, vs = [x[at:at + n] for x in kl], [x[at:at + n] for x in vl]
            enl.enl_group_store_all_layers(state.cache, first + i, ks, vs, stream=stream)
            if first + i in state.keep:
                rows[first + i] = ([x.clone() for x in ks], [x.clone() for x in vs])
            if evict:
                enl.enl_group_evict(state.cache, first + i, stream=stream)
            at += n
    return rows


def _cu(parts):
    return np.concatenate([[0], np.cumsum(parts)]).astype(np.int32)


def prepare(case, seed):
    s, kind, layers = _shapes(case), case["kind"], case["layers"]
    hq, hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    st = State(case)

    if kind == "static":
        n = int(s["seg_len"].sum()) + case["new"]
        st.seg_len, st.q = s["seg_len"].astype(np.int32), _per_layer(_queries(gen, case, 1).squeeze(1))
        st.k, st.v = _per_layer(_rows(gen, layers, n, hkv, d)), _per_layer(_rows(gen, layers, n, hkv, d))
        st.out = torch.zeros(layers, hq, d, dtype=BF16, device="cuda")
        st.mass = torch.zeros(layers, hq, case["segs"] + 1, device="cuda") if case["mass"] else None
        st.outs, st.masses = _per_layer(st.out), _per_layer(st.mass) if case["mass"] else [None] * layers
        return st

    if kind == "update":
        st.keep = set(s["touched"])
        n_q = max(s["add"])
        rows = _fill(case, st, gen, s["lens"], 1, n_q, extra=sum(s["add"]))
        st.jobs, st.outs = [], []
        for g, n in zip(s["touched"], s["add"]):
            job = dict(group=g, n=n, base=rows[g], sel=np.array([g], np.int32))
            for name, heads, sigma in (("q", hq, SCORE_STD), ("k", hkv, 1.0), ("v", hkv, 1.0)):
                job[name + "_new"] = _rows(gen, layers, n, heads, d, sigma)                # as the projections leave them
                job[name] = job[name + "_new"].clone()
                job[name + "_layers"] = _per_layer(job[name])
            job["pos"] = (int(s["lens"][0][g]) + torch.arange(n, dtype=torch.int32, device="cuda")).repeat(layers)
            st.outs.append(torch.zeros(layers, n, hq, d, dtype=BF16, device="cuda"))
            job["out"] = _per_layer(st.outs[-1])
            st.jobs.append(job)
        # one query over the whole map: what the next token sees of the update
        st.sel = np.arange(case["groups"], dtype=np.int32)
        st.q, st.kn, st.vn = (_per_layer(_rows(gen, layers, 1, h, d, x)) for h, x in ((hq, SCORE_STD), (hkv, 1.0), (hkv, 1.0)))
        st.outs.append(torch.zeros(layers, 1, hq, d, dtype=BF16, device="cuda"))
        st.out = _per_layer(st.outs[-1])
        return st

    if kind == "tier":
        st.keep = set()
        st.lists = [(p, s["mem"]) for p in s["prob"]]
        # device pages for one step's choice and hardly more (the library adds a page per group to the tokens asked for)
        pages = max(int((-(-s["lens"][0][c] // 16)).sum()) for c in s["chosen"]) + -(-case["len_hi"] // 16)
        _fill(case, st, gen, s["lens"], 1, case["n_q"], capacity=max(16, 16 * (pages - case["groups"])), evict=True)
        st.q = _per_layer(_queries(gen, case, case["n_q"]))
        st.kn, st.vn = (_per_layer(_rows(gen, layers, case["n_q"], hkv, d)) for _ in range(2))
        st.out = torch.zeros(2, layers, case["n_q"], hq, d, dtype=BF16, device="cuda")
        st.outs = [_per_layer(x) for x in st.out]
        st.s = s
        return st

    # plan, score, decode: a filled map and the select list of the step
    base = np.cumsum([0] + [len(x) for x in s["lens"]])
    st.sel = np.concatenate([b + x for b, x in zip(base, s["sel"])]).astype(np.int32)
    batch = len(s["lens"])
    many = batch > 1
    cu_sel = _cu([len(x) for x in s["sel"]]) if many else None
    slots = max(len(x) for x in s["sel"]) + 1

    if kind == "decode":
        st.keep = set()
        _fill(case, st, gen, s["lens"], batch, batch)
        last = [n + case["tokens"] - 1 for n in s["n_new"]]
        grown = [(_rows(gen, layers, n, hkv, d), _rows(gen, layers, n, hkv, d)) for n in last]
        st.steps = []
        st.out = torch.zeros(case["tokens"], layers, batch, hq, d, dtype=BF16, device="cuda")
        st.mass = torch.zeros(case["tokens"], layers, batch, hq, slots, device="cuda") if case["mass"] else None
        for j in range(case["tokens"]):
            seen = [n + j for n in s["n_new"]]
            if many:                                            # the episodes' rows lie back to back
                k, v = (torch.cat([g[i][:, :n] for g, n in zip(grown, seen)], dim=1) for i in (0, 1))
            else:                                               # one episode: the buffer that the decoding fills
                k, v = grown[0]
            st.steps.append(dict(q=_per_layer(_queries(gen, case, batch)), k=_per_layer(k), v=_per_layer(v), n_new=sum(seen),
                                 out=_per_layer(st.out[j]), mass=_per_layer(st.mass[j]) if case["mass"] else [None] * layers,
                                 cu_sel=cu_sel, cu_q=_cu([1] * batch) if many else None, cu_new=_cu(seen) if many else None))
        return st

    n_q, n_new = sum(s["n_q"]), sum(s["n_new"])
    st.group = int(st.sel[0])
    st.keep = {st.group}
    q = _queries(gen, case, n_q)
    affinity = None
    if kind == "score":                                         # an object's queries lean towards its group's keys
        a = math.sqrt(4.0 / math.sqrt(d))
        affinity = _randn(gen, (case["groups"], hkv, d), a)
        lean = torch.zeros(n_q, hq, d, dtype=BF16, device="cuda")
        for o, t in enumerate(s["target"]):
            if t >= 0:
                lean[s["obj_off"][o]:s["obj_off"][o + 1]] = affinity[int(t)].repeat_interleave(hq // hkv, dim=0)
        q += lean
    st.base = _fill(case, st, gen, s["lens"], batch, n_q, affinity=affinity)[st.group]
    st.q = _per_layer(q)
    st.kn, st.vn = (_per_layer(_rows(gen, layers, n_new, hkv, d)) for _ in range(2))
    if kind == "score":
        n_obj = len(s["obj_off"]) - 1
        st.obj_off, st.threshold = s["obj_off"], 5.0 / case["groups"]
        kept = 1 if case["sums"] else layers
        st.mass = torch.zeros(kept, n_q, hq, slots, device="cuda")
        st.masses = _per_layer(st.mass)
        st.out = None if case["sums"] else torch.zeros(layers, n_q, hq, d, dtype=BF16, device="cuda")
        st.sums = torch.zeros(n_obj, slots, device="cuda") if case["sums"] else None
        st.avg = torch.zeros(n_obj, case["groups"], device="cuda")
        st.assign = torch.zeros(n_obj, dtype=torch.int32, device="cuda")
    else:
        st.cu_sel, st.cu_q, st.cu_new = (cu_sel, _cu(s["n_q"]), _cu(s["n_new"])) if many else (None, None, None)
        st.out = torch.zeros(layers, n_q, hq, d, dtype=BF16, device="cuda")
        st.mass = torch.zeros(layers, n_q, hq, slots, device="cuda") if case["mass"] else None
        st.masses = _per_layer(st.mass) if case["mass"] else [None] * layers
    st.outs = _per_layer(st.out) if st.out is not None else None
    return st


# ---- one pass -----------------------------------------------------------------------------------------------------
def _plan(st, stream):
    enl.enl_group_store_all_layers(st.cache, st.group, st.base[0], st.base[1], stream=stream)
    for layer in range(st.case["layers"]):
        enl.enl_attend(st.cache, layer, st.sel, st.q[layer], st.kn[layer], st.vn[layer], st.outs[layer], st.masses[layer],
                       cu_sel=st.cu_sel, cu_q=st.cu_q, cu_new=st.cu_new, stream=stream)
    return {"out": st.out, "mass": st.mass}


def _score(st, stream):
    case = st.case
    enl.enl_group_store_all_layers(st.cache, st.group, st.base[0], st.base[1], stream=stream)
    if not case["sums"]:
        for layer in range(case["layers"]):
            enl.enl_attend(st.cache, layer, st.sel, st.q[layer], st.kn[layer], st.vn[layer], st.outs[layer], st.masses[layer],
                           stream=stream)
        enl.enl_cluster_assign(st.masses, st.obj_off, case["groups"], st.threshold, st.avg, st.assign, stream=stream)
        return {"out": st.out, "mass": st.mass, "avg": st.avg, "assign": st.assign}
    st.sums.zero_()
    for layer in range(case["layers"]):
        enl.enl_attend(st.cache, layer, st.sel, st.q[layer], st.kn[layer], st.vn[layer], None, st.masses[0],
                       flags=enl.ENL_MASS_ONLY, group_mass_sum=st.sums, obj_off=st.obj_off, stream=stream)
    enl.enl_cluster_assign_sums(st.sums, st.obj_off, case["groups"], case["q_heads"], case["layers"], st.threshold, st.avg,
                                st.assign, stream=stream)
    return {"mass": st.mass, "sums": st.sums, "avg": st.avg, "assign": st.assign}


def _decode(st, stream):
    for t in st.steps:
        for layer in range(st.case["layers"]):
            enl.enl_attend(st.cache, layer, st.sel, t["q"][layer], t["k"][layer], t["v"][layer], t["out"][layer], t["mass"][layer],
                           cu_sel=t["cu_sel"], cu_q=t["cu_q"], cu_new=t["cu_new"], n_new=t["n_new"], stream=stream)
    return {"out": st.out, "mass": st.mass}


def _update(st, stream):
    layers = st.case["layers"]
    for job in st.jobs:
        if st.case["per_layer"]:
            for layer in range(layers):
                enl.enl_group_store(st.cache, job["group"], layer, job["base"][0][layer], job["base"][1][layer], stream=stream)
        else:
            enl.enl_group_store_all_layers(st.cache, job["group"], job["base"][0], job["base"][1], stream=stream)
        for name in ("q", "k"):
            job[name].copy_(job[name + "_new"])
            enl.enl_rope_rotate(job[name].view(-1, *job[name].shape[2:]), positions=job["pos"], stream=stream)
        for layer in range(layers):
            enl.enl_attend(st.cache, layer, job["sel"], job["q_layers"][layer], job["k_layers"][layer], job["v_layers"][layer],
                           job["out"][layer], stream=stream)
        if st.case["per_layer"]:
            for layer in range(layers):
                enl.enl_group_store(st.cache, job["group"], layer, job["k_layers"][layer], job["v_layers"][layer],
                                    mode=enl.ENL_APPEND, stream=stream)
        else:
            enl.enl_group_store_all_layers(st.cache, job["group"], job["k_layers"], job["v_layers"], mode=enl.ENL_APPEND,
                                           stream=stream)
    for layer in range(layers):
        enl.enl_attend(st.cache, layer, st.sel, st.q[layer], st.kn[layer], st.vn[layer], st.out[layer], stream=stream)
    return {"out": st.outs}


def _tier(st, stream):
    s, picked = st.s, []
    for (prob, mem), outs in zip(st.lists, st.outs):
        sel = enl.enl_select_knapsack(prob, s["threshold"], mem, s["budget"], s["quantum"])
        enl.enl_step_prepare(st.cache, sel, stream=stream)
        for layer in range(st.case["layers"]):
            enl.enl_attend(st.cache, layer, sel, st.q[layer], st.kn[layer], st.vn[layer], outs[layer], stream=stream)
        picked.append(sel)
    return {"out": st.out, "picked": picked}


def _static(st, stream):
    for layer in range(st.case["layers"]):
        enl.enl_attend_static(st.seg_len, st.case["new"], st.q[layer], st.k[layer], st.v[layer], st.outs[layer], st.masses[layer],
                              stream=stream)
    return {"out": st.out, "mass": st.mass}


_RUN = {"plan": _plan, "score": _score, "decode": _decode, "update": _update, "tier": _tier, "static": _static}


def run(state):
    return _RUN[state.case["kind"]](state, torch.cuda.current_stream().cuda_stream)
