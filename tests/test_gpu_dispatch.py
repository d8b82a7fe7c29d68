"""GPU parity at the sizes where the library goes from one way of doing a call to another, against the float64 oracle."""
import numpy as np
import pytest
import torch

from oracle import enl_oracle as orc
from paper_2510_18546_b200 import enl, synth
from tests.helpers import Session, check_close

pytestmark = pytest.mark.gpu


def check(wl, rows=None, **kw):
    """Layer 0 of a one-episode workload against the oracle (some rows of it, or all)."""
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        out, mass, _ = s.attend(0, q, kn, vn, **kw)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        ro, rm, _ = s.oracle(0, 0, q, kn, vn, rows=rows)
        pick = slice(None) if rows is None else torch.tensor(rows, device=q.device)
        check_close(out[pick], ro, None if mass is None else mass[pick], rm if mass is not None else None, what=wl.name)


@pytest.mark.parametrize("pages", [200, 232, 260, 990, 1030, 3520, 3640])
@pytest.mark.parametrize("n_q", [1, 40])
def test_gather_plan_reaches_the_device(pages, n_q):
    """Plans on either side of the sizes that travel as launch parameters (2, 8 and 28 KB) and of the copied one; two
    calls with different lists in a row, so that the second plan replaces the first one while that is in use."""
    lens = [160] * (pages // 10) + [16] * (pages % 10)
    wl = synth.make_small(31, 1, 4, 1, 64, [lens], [list(range(len(lens)))], [n_q], [n_q], name=f"plan {pages} pages")
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        short = np.arange(len(lens) // 2, dtype=np.int32)
        outs = []
        for sel in (short, wl.sel_ids()):
            out = torch.empty_like(q)
            mass = torch.empty(n_q, 4, len(sel) + 1, device=s.device)
            enl.enl_attend(s.cache, 0, sel, q, kn, vn, out, mass)
            outs.append((out, mass, sel))
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        rows = [0, n_q - 1] if n_q > 1 else [0]
        for out, mass, sel in outs:
            ks, vs = ([x[i] for i in sel] for x in s.host_kv[(0, 0)])
            ro, rm = orc.attend_slots(4, 1, 64, ks, vs, q.cpu(), kn.cpu(), vn.cpu(), rows=rows)
            check_close(out[rows], ro, mass[rows], rm, what=f"{wl.name}, {len(sel)} groups")


# One-token steps merged by clusters: slots that reach over several CTAs' ranges, ranges that begin and end on slot
# boundaries, empty groups, more slots than pages in a range, every number of q heads per kv head, streams from one page up to
# where the streaming kernel takes over.
STEP = {
    "one_page": dict(Hq=4, Hkv=1, D=128, pool=[[10]], sel=[[]], n_new=[3]),
    "two_pages": dict(Hq=2, Hkv=2, D=64, pool=[[5]], n_new=[1]),
    "sixteen_pages": dict(Hq=8, Hkv=2, D=128, pool=[[16] * 8], n_new=[128]),
    "one_slot_over_all_ranges": dict(Hq=8, Hkv=1, D=128, pool=[[3000]], n_new=[1]),
    "slots_of_one_key": dict(Hq=16, Hkv=8, D=64, pool=[[1] * 200], n_new=[17]),
    "empty_groups": dict(Hq=4, Hkv=4, D=128, pool=[[0, 0, 300, 0, 17, 0, 0]], n_new=[40]),
    "long_new": dict(Hq=32, Hkv=8, D=128, pool=[[90, 33]], n_new=[700]),
    "below_the_line": dict(Hq=32, Hkv=8, D=128, pool=[[1008 * 16 // 4] * 4], n_new=[16]),
    "above_the_line": dict(Hq=32, Hkv=8, D=128, pool=[[1032 * 16 // 4] * 4], n_new=[16]),
    "batch": dict(Hq=8, Hkv=2, D=128, pool=[[30, 60, 90], [5, 5, 5, 5], [200], [], [700, 1]], n_new=[1, 10, 129, 16, 33]),
    "eights_at_most": dict(Hq=32, Hkv=8, D=128, pool=[[90 * 16 // 4] * 4], n_new=[96]),
    "eights_with_masses": dict(Hq=32, Hkv=8, D=128, pool=[[47 * 16] * 4], n_new=[64]),
    "sixteens_again": dict(Hq=32, Hkv=8, D=128, pool=[[48 * 16] * 4], n_new=[16]),
    "many_clusters": dict(Hq=16, Hkv=8, D=64, pool=[[40, 25]] * 20, n_new=[9] * 20),
}


@pytest.mark.parametrize("want_mass", [True, False])
@pytest.mark.parametrize("name", sorted(STEP))
def test_one_token_steps(name, want_mass):
    c = STEP[name]
    n = len(c["pool"])
    wl = synth.make_small(41, 1, c["Hq"], c["Hkv"], c["D"], c["pool"],
                          c.get("sel") or [list(range(len(x)))[::-1] for x in c["pool"]], [1] * n, c["n_new"], name=name)
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        cn = wl.cu()[2]
        for _ in range(2):                                  # the second call finds plan and pool as the first left them
            out, mass, _ = s.attend(0, q, kn, vn, want_mass=want_mass)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        for b in range(n):
            ro, rm, _ = s.oracle(0, b, q[b:b + 1], kn[cn[b]:cn[b + 1]], vn[cn[b]:cn[b + 1]])
            G = len(wl.sel_local[b])
            check_close(out[b:b + 1], ro, mass[b:b + 1, :, :G + 1] if want_mass else None, rm if want_mass else None, what=name)


def test_stores_between_one_token_steps_are_seen():
    """A store directly before a step, and steps directly after one another: what may be read before the previous launch has
    ended is exactly what no launch in between has written."""
    wl = synth.make_small(43, 1, 8, 2, 128, [[60, 90, 33]], [[0, 1, 2]], [1], [1], name="store between steps")
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        k, v = wl.pool_kv(0, 0, s.device)
        outs, want = [], []
        gen = torch.Generator(device=s.device).manual_seed(5)
        for i in range(6):
            if i % 2 == 0:
                k[60:150] = torch.randn(90, 2, 128, generator=gen, device=s.device).to(k.dtype)
                rows = k[60:150].clone()
                enl.enl_group_store(s.cache, 1, 0, rows, v[60:150])
            out = torch.empty_like(q)
            enl.enl_attend(s.cache, 0, [0, 1, 2], q, kn, vn, out)
            outs.append(out)
            ks = [k[a:b].cpu().clone() for a, b in ((0, 60), (60, 150), (150, 183))]
            vs = [v[a:b].cpu() for a, b in ((0, 60), (60, 150), (150, 183))]
            want.append((ks, vs))
        torch.cuda.synchronize()
        for out, (ks, vs) in zip(outs, want):
            ro, _ = orc.attend_slots(8, 2, 128, ks, vs, q.cpu(), kn.cpu(), vn.cpu())
            check_close(out, ro, None, None, what="store between steps")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("rep", [1, 2, 8])
@pytest.mark.parametrize("lens, n_new", [([], 1), ([0, 5, 0, 0, 16, 1], 1), ([1] * 255, 2), ([700, 15, 17], 33), ([40000], 9)])
@pytest.mark.parametrize("shift", [0, 1])
def test_static_step(D, rep, lens, n_new, shift):
    """Segments that start anywhere; with shift the tensors start off a 16-byte boundary (the other kernel)."""
    if shift and sum(lens) > 10000:
        pytest.skip("one long stream is enough")
    hkv = 2
    n = sum(lens) + n_new
    gen = torch.Generator(device="cuda").manual_seed(n)

    def rand(*shape):
        x = torch.randn(int(np.prod(shape)) + shift, generator=gen, device="cuda").to(torch.bfloat16)
        return x[shift:].view(*shape)

    q, k, v = rand(hkv * rep, D), rand(n, hkv, D), rand(n, hkv, D)
    out = torch.full_like(q, float("nan"))
    mass = torch.full((hkv * rep, len(lens) + 1), float("nan"), device="cuda")
    enl.enl_attend_static(lens, n_new, q, k, v, out, mass)
    torch.cuda.synchronize()
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(int)
    ks, vs = ([x[a:b].cpu() for a, b in zip(offs[:-1], offs[1:])] for x in (k, v))
    ro, rm = orc.attend_slots(hkv * rep, hkv, D, ks, vs, q[None].cpu(), k[offs[-1]:].cpu(), v[offs[-1]:].cpu())
    check_close(out[None], ro, mass[None], rm, what="static")


# Masses without outputs: slots that end anywhere in a key tile, that reach over several splits, one Q tile and two, rows at
# the causal limit, scores that jump by hundreds between tiles.
MASS = {
    "one_tile": dict(Hq=4, Hkv=1, D=128, pool=[[5, 16, 1]], n_q=[7], n_new=[7]),
    "ragged": dict(Hq=8, Hkv=2, D=128, pool=[[1, 50, 16, 33, 7, 120, 15, 17, 300]], n_q=[77], n_new=[200]),
    "slot_over_all_splits": dict(Hq=4, Hkv=2, D=64, pool=[[20, 2500, 3]], n_q=[130], n_new=[130]),
    "many_slots": dict(Hq=8, Hkv=8, D=128, pool=[[1 + i % 9 for i in range(300)]], n_q=[129], n_new=[129]),
    "batch": dict(Hq=16, Hkv=2, D=128, pool=[[30, 0, 90], [700, 5, 250], [200]], n_q=[70, 3, 129], n_new=[70, 10, 129]),
}


@pytest.mark.parametrize("split", [0, 1, 3, 8])
@pytest.mark.parametrize("name", sorted(MASS))
def test_masses_without_outputs(name, split):
    c = MASS[name]
    n = len(c["pool"])
    wl = synth.make_small(47, 1, c["Hq"], c["Hkv"], c["D"], c["pool"], [list(range(len(x)))[::-1] for x in c["pool"]], c["n_q"],
                          c["n_new"], name=name)
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        if name == "ragged":
            q = (q.float() * torch.linspace(1, 40, q.shape[0], device=s.device)[:, None, None]).to(q.dtype)
        cs, cq, cn = wl.cu()
        G = max(len(x) for x in wl.sel_local)
        mass = torch.full((q.shape[0], wl.n_q_heads, G + 1), float("nan"), device=s.device)
        enl.enl_attend(s.cache, 0, wl.sel_ids(), q, kn, vn, None, mass, cu_sel=cs if n > 1 else None, cu_q=cq if n > 1 else None,
                       cu_new=cn if n > 1 else None, split_hint=split, flags=enl.ENL_MASS_ONLY)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        for b in range(n):
            rows = sorted({0, c["n_q"][b] // 2, c["n_q"][b] - 1, min(63, c["n_q"][b] - 1)})
            _, rm, _ = s.oracle(0, b, q[cq[b]:cq[b + 1]], kn[cn[b]:cn[b + 1]], vn[cn[b]:cn[b + 1]], rows=rows)
            g = len(wl.sel_local[b])
            got = mass[cq[b]:cq[b + 1]][rows, :, :g + 1].cpu().numpy()
            assert np.abs(got - rm).max() < 1e-4, f"{name} episode {b}"


# Short calls: rows at the edges of a CTA's 64, key streams up to the 24 pages that stay resident and one beyond, empty lists and groups, every number
# of q heads per kv head, episodes of different sizes, queries that are only the last of the new tokens.
SHORT = {
    "one_row_pair": dict(Hq=2, Hkv=2, D=64, pool=[[3]], sel=[[0]], n_q=[2], n_new=[2]),
    "rows_63": dict(Hq=2, Hkv=2, D=128, pool=[[40, 17]], sel=[[1, 0]], n_q=[63], n_new=[63]),
    "rows_64": dict(Hq=8, Hkv=2, D=128, pool=[[40, 17]], sel=[[0, 1]], n_q=[16], n_new=[16]),
    "rows_65": dict(Hq=1, Hkv=1, D=64, pool=[[40, 17]], sel=[[0, 1]], n_q=[65], n_new=[65]),
    "rep16": dict(Hq=32, Hkv=2, D=128, pool=[[33, 50]], sel=[[0, 1]], n_q=[9], n_new=[9]),
    "rep8": dict(Hq=32, Hkv=4, D=64, pool=[[33, 50]], sel=[[0, 1]], n_q=[41], n_new=[41]),
    "pages_24": dict(Hq=32, Hkv=8, D=128, pool=[[160, 128]], sel=[[0, 1]], n_q=[61], n_new=[96]),
    "pages_25": dict(Hq=32, Hkv=8, D=128, pool=[[160, 128]], sel=[[0, 1]], n_q=[61], n_new=[97]),
    "slots_as_pages": dict(Hq=8, Hkv=2, D=128, pool=[[1] * 20], sel=[list(range(20))], n_q=[30], n_new=[30]),
    "empty_select": dict(Hq=8, Hkv=2, D=128, pool=[[10]], sel=[[]], n_q=[100], n_new=[100]),
    "empty_groups": dict(Hq=8, Hkv=2, D=64, pool=[[0, 0, 40, 0, 5, 0]], sel=[[0, 1, 2, 3, 4, 5]], n_q=[20], n_new=[20]),
    "prior": dict(Hq=8, Hkv=2, D=128, pool=[[30]], sel=[[0]], n_q=[5], n_new=[200]),
    "batch": dict(Hq=8, Hkv=2, D=128, pool=[[30, 60, 90], [5, 5, 5, 5], [200]], sel=[[2, 0], [0, 1, 2, 3], []],
                  n_q=[70, 3, 129], n_new=[70, 10, 129]),
}


@pytest.mark.parametrize("want_mass", [True, False])
@pytest.mark.parametrize("name", sorted(SHORT))
def test_short_calls(name, want_mass):
    c = SHORT[name]
    wl = synth.make_small(53, 1, c["Hq"], c["Hkv"], c["D"], c["pool"], c["sel"], c["n_q"], c["n_new"], name=name)
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        q = q * 3
        _, cq, cn = wl.cu()
        for _ in range(2):                                  # the second call finds plan and pool as the first left them
            out, mass, _ = s.attend(0, q, kn, vn, want_mass=want_mass)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        for b in range(wl.batch):
            ro, rm, _ = s.oracle(0, b, q[cq[b]:cq[b + 1]], kn[cn[b]:cn[b + 1]], vn[cn[b]:cn[b + 1]])
            G = len(wl.sel_local[b])
            check_close(out[cq[b]:cq[b + 1]], ro, mass[cq[b]:cq[b + 1], :, :G + 1] if want_mass else None, rm if want_mass else None, what=name)


@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("heads, D, n", [(32, 128, 5), (8, 128, 5), (1, 16, 9), (3, 48, 7), (2, 256, 3), (2, 24, 6), (40, 256, 2)])
def test_rope_pieces(heads, D, n, interleaved):
    """Sizes around the rows and heads that a CTA takes, and head sizes that do not split into 16-byte pieces."""
    gen = torch.Generator(device="cuda").manual_seed(D)
    x = torch.randn(n, heads, D, generator=gen, device="cuda").to(torch.bfloat16)
    pos = torch.tensor([(i * 7919) % 120_000 for i in range(n)], dtype=torch.int32, device="cuda")
    want = orc.rope_rotate(x.float().cpu().numpy(), pos.cpu().numpy(), 10000.0, interleaved)
    got = x.clone()
    enl.enl_rope_rotate(got, positions=pos, interleaved=interleaved)
    torch.cuda.synchronize()
    err = np.abs(got.float().cpu().numpy() - want)
    assert (err <= np.maximum(np.abs(want) * 2.0 ** -8, 1e-4)).all(), err.max()


@pytest.mark.parametrize("splits", [0, 3, 4, 5, 8, 9, 17])
@pytest.mark.parametrize("n_q", [40, 150])
def test_splits_and_ragged_pages(n_q, splits):
    """Merging up to four, eight and more splits (0: as many as the library likes), more than 32 slots, and groups of 1 to 45
    tokens, so that pages of every fill stand in the key tiles."""
    lens = list(range(1, 46))
    wl = synth.make_small(61, 1, 8, 2, 128, [lens + [700, 800]], [list(range(47))[::-1]], [n_q], [n_q], name=f"{splits} splits")
    check(wl, split_hint=splits)


@pytest.mark.parametrize("slots", [24, 25, 26, 27])
def test_slots_parked_in_shared_memory(slots):
    wl = synth.make_small(62, 1, 8, 2, 128, [[30] * (slots - 1)], [list(range(slots - 1))], [300], [300], name=f"{slots} slots")
    check(wl, rows=[0, 127, 128, 299])


@pytest.mark.parametrize("pages", [3, 17, 33, 70])
def test_loads_beside_the_stream(pages):
    """Loads of one chunk and of chunks of several layers and of one (64 KB per page and layer, 2 MB per chunk): layers in any
    order right behind the load, another stream, a captured graph, a store and an eviction that overtake nothing."""
    L, half = 5, pages * 8 + 5                              # the two groups of a list fill `pages` pages, and one more
    wl = synth.make_small(63, L, 8, 8, 128, [[half] * 4], [[0, 1]], [20], [20], name=f"load {pages} pages")
    with Session(wl, list(range(L)), extra_tokens=64) as s:
        enl.enl_tier_enable(s.cache, 8 * half)
        q, kn, vn = wl.new_qkv(0, s.device)

        def attend(sel, layer, stream=None):
            out = torch.empty_like(q)
            enl.enl_attend(s.cache, layer, sel, q, kn, vn, out, stream=torch.cuda.current_stream().cuda_stream if stream is None else stream)
            return out

        def swap(i):                                        # the other list out, this one in
            for g in sels[1 - i]:
                enl.enl_group_evict(s.cache, g)
            enl.enl_step_prepare(s.cache, sels[i])

        sels = ([0, 1], [2, 3])
        want = [[attend(sel, l) for l in range(L)] for sel in sels]
        torch.cuda.synchronize()
        for i in (0, 1, 0):
            swap(i)
            got = {l: attend(sels[i], l) for l in (4, 0, 2, 1, 3)}
            torch.cuda.synchronize()
            assert all(torch.equal(got[l], want[i][l]) for l in range(L))
        swap(1)
        swap(0)                                             # nothing has waited for the load before
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        out = attend(sels[0], 4, stream=side.cuda_stream)
        torch.cuda.synchronize()
        assert torch.equal(out, want[0][4])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = attend(sels[0], 3)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want[0][3])
        rows = torch.zeros(half, 8, 128, device=s.device, dtype=torch.bfloat16)
        swap(1)
        swap(0)
        for l in range(L):                                  # over what has just been loaded
            enl.enl_group_store(s.cache, 0, l, rows, rows)
        got = [attend([0], l) for l in range(L)]
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        zero = rows.cpu()
        ro, _ = orc.attend_slots(8, 8, 128, [zero], [zero], q.cpu(), kn.cpu(), vn.cpu())
        for out in got:
            check_close(out, ro, None, None, what=wl.name)


def test_short_calls_between_long_ones_and_stores():
    """A short call takes its pages along, a long one reads them from device memory: either after the other and after a store."""
    wl = synth.make_small(64, 1, 8, 2, 128, [[40, 30, 600]], [[0, 1, 2]], [20], [20], name="short and long in turn")
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        k, v = wl.pool_kv(0, 0, s.device)
        gen = torch.Generator(device=s.device).manual_seed(6)
        spans, outs, want = ((0, 40), (40, 70), (70, 670)), [], []
        for i in range(8):
            if i % 3 == 0:
                k[:40] = torch.randn(40, 2, 128, generator=gen, device=s.device).to(k.dtype)
                enl.enl_group_store(s.cache, 0, 0, k[:40].clone(), v[:40])
            sel = ([0, 1], [0, 2], [1, 0], [2, 0])[i % 4]
            out = torch.empty_like(q)
            enl.enl_attend(s.cache, 0, sel, q, kn, vn, out)
            outs.append(out)
            want.append([[x[a:b].cpu().clone() for a, b in (spans[g] for g in sel)] for x in (k, v)])
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        for out, (ks, vs) in zip(outs, want):
            ro, _ = orc.attend_slots(8, 2, 128, ks, vs, q.cpu(), kn.cpu(), vn.cpu())
            check_close(out, ro, None, None, what=wl.name)


@pytest.mark.parametrize("n_q, pages", [(20, 4), (300, 60), (1, 60), (40, 3700)])
def test_graphs_and_calls_beside_them(n_q, pages):
    """A call captured into a graph that has not run yet, calls outside the graph before and after it runs, over either list: each
    goes by its own gather plan (in the parameters, written in one piece, in several)."""
    wl = synth.make_small(65, 1, 4, 1, 64, [[5, 40, 16 * pages]], [[0, 1, 2]], [n_q], [n_q], name=f"graph {n_q} rows, {pages} pages")
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        lists = [np.asarray(x, np.int32) for x in ([2, 0], [1, 2])]

        def attend(i):
            out = torch.empty_like(q)
            enl.enl_attend(s.cache, 0, lists[i], q, kn, vn, out, stream=torch.cuda.current_stream().cuda_stream)
            return out

        got = [(0, attend(0))]
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            in_graph = attend(1)
        got += [(1, attend(1)), (0, attend(0))]
        graph.replay()
        got += [(0, attend(0)), (1, in_graph.clone()), (1, attend(1))]
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        rows = sorted({0, n_q // 2, n_q - 1})
        for i, out in got:
            ks, vs = ([x[g] for g in lists[i]] for x in s.host_kv[(0, 0)])
            ro, _ = orc.attend_slots(4, 1, 64, ks, vs, q.cpu(), kn.cpu(), vn.cpu(), rows=rows)
            check_close(out[rows], ro, None, None, what=f"{wl.name}, list {i}")


@pytest.mark.parametrize("n_q", [1, 20, 300])
def test_captured_stores_are_seen_by_calls_outside_the_graph(n_q):
    """A graph that stores runs before, between and directly in front of calls outside it, with other rows every time: each call sees what
    the graph has written last."""
    lens = [64, 200, 48]
    wl = synth.make_small(66, 1, 8, 2, 128, [lens], [[0, 1, 2]], [n_q], [n_q], name=f"captured store, {n_q} rows")
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        k, v = (x.clone() for x in wl.pool_kv(0, 0, s.device))
        rows_k, rows_v = k[64:264].clone(), v[64:264].clone()

        def attend():
            out = torch.empty_like(q)
            enl.enl_attend(s.cache, 0, [0, 1, 2], q, kn, vn, out, stream=torch.cuda.current_stream().cuda_stream)
            return out

        attend()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            enl.enl_group_store(s.cache, 1, 0, rows_k, rows_v, stream=torch.cuda.current_stream().cuda_stream)
        gen = torch.Generator(device=s.device).manual_seed(7)
        got = []
        for _ in range(4):
            for _ in range(2):                          # launches that nothing has been written between
                attend()
            rows_k.copy_(torch.randn(200, 2, 128, generator=gen, device=s.device))
            graph.replay()
            got.append((rows_k.cpu(), attend(), attend()))
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        rows = sorted({0, n_q // 2, n_q - 1})
        for now, *outs in got:
            ks = [k[:64].cpu(), now, k[264:].cpu()]
            vs = [v[:64].cpu(), v[64:264].cpu(), v[264:].cpu()]
            ro, _ = orc.attend_slots(8, 2, 128, ks, vs, q.cpu(), kn.cpu(), vn.cpu(), rows=rows)
            for out in outs:
                check_close(out[rows], ro, None, None, what=wl.name)


@pytest.mark.parametrize("splits", [3, 5, 33, 40])
@pytest.mark.parametrize("groups", [25, 31, 32, 63, 64, 65, 130])
def test_masses_of_splits_merged_in_memory(groups, splits):
    """More slots than fit shared memory, each in one or two of the splits: the merge takes them from where the splits have walked them, 64 at a
    time.  The scratch buffer holds another call's partial results, so slots that a split has not written are anything."""
    lens = [max(1, 2 * 5400 // groups * (1 + i % 3) // 4) for i in range(groups)]
    lens[groups // 2] = 0
    wl = synth.make_small(67, 1, 4, 1, 64, [lens], [list(range(groups))], [40], [50], name=f"{groups} groups in {splits} splits")
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        s.attend(0, q * 3, kn, vn, split_hint=splits, sel_override=list(range(groups))[::-1])
        out, mass, _ = s.attend(0, q, kn, vn, split_hint=splits)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        p = enl.enl_plan_inspect(s.cache)
        assert p["n_splits"] == splits and p["merge_kind"] == 1
        ro, rm, _ = s.oracle(0, 0, q, kn, vn)
        check_close(out, ro, mass, rm, what=wl.name)
