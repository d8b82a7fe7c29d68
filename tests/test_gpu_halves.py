"""Prefill calls with few CTAs: a Q tile per CTA whose key steps its two walkers share.  Where the halves meet (inside a group, between two,
at an empty one, in the new tokens), odd numbers of steps, one row to several tiles, with and without splits on top (`splits`), slots that
fit shared memory and more.  (That these calls are planned as such is checked without a GPU, in test_host_state.py.)"""
import numpy as np
import pytest
import torch

from paper_2510_18546_b200 import enl, synth
from tests.helpers import Session, check_close

pytestmark = pytest.mark.gpu

CASES = {
    "meet_inside_a_group": dict(Hq=8, Hkv=2, D=128, pool=[[30, 500, 20]], n_q=[70], n_new=[70], splits=True),
    "meet_between_groups": dict(Hq=8, Hkv=2, D=128, pool=[[256, 256]], n_q=[40], n_new=[40], splits=True),
    "meet_at_an_empty_group": dict(Hq=8, Hkv=2, D=128, pool=[[240, 0, 0, 224]], n_q=[40], n_new=[40], splits=True),
    "meet_in_the_new_tokens": dict(Hq=8, Hkv=2, D=128, pool=[[100]], n_q=[400], n_new=[400], splits=False),
    "slots_in_the_mass_buffer": dict(Hq=8, Hkv=2, D=128, pool=[[5 + (i * 7) % 23 for i in range(40)]], n_q=[100], n_new=[100], splits=True),
    "rows_of_one_tile": dict(Hq=32, Hkv=8, D=128, pool=[[3000, 33]], n_q=[17], n_new=[17], splits=True),
    "one_row_beyond_a_tile": dict(Hq=32, Hkv=8, D=128, pool=[[400, 33, 7]], n_q=[33], n_new=[95], splits=True),
    "odd_steps_d64": dict(Hq=8, Hkv=2, D=64, pool=[[64 * 7]], n_q=[65], n_new=[65], splits=True),
    "rep1": dict(Hq=2, Hkv=2, D=64, pool=[[300, 200]], n_q=[140], n_new=[140], splits=True),
    "rep8_long": dict(Hq=8, Hkv=1, D=128, pool=[[2000, 45, 1100]], n_q=[40], n_new=[40], splits=True),
    "unsplit_inside_a_group": dict(Hq=32, Hkv=8, D=128, pool=[[30, 500, 20]], n_q=[310], n_new=[310], splits=False),
    "unsplit_d64": dict(Hq=16, Hkv=16, D=64, pool=[[100, 77, 200]], n_q=[600], n_new=[650], splits=False),
    "unsplit_slots_in_the_mass_buffer": dict(Hq=32, Hkv=8, D=128, pool=[[5 + (i * 7) % 23 for i in range(40)]], n_q=[310], n_new=[310], splits=False),
    "unsplit_ends_in_the_mass_buffer": dict(Hq=32, Hkv=8, D=128, pool=[[16] * 60], n_q=[297], n_new=[300], splits=False),
    "batch": dict(Hq=8, Hkv=2, D=128, pool=[[300, 60, 90], [5, 5, 450], [400]], n_q=[70, 3, 129], n_new=[70, 10, 129], splits=True),
}


@pytest.mark.parametrize("want_mass", [True, False])
@pytest.mark.parametrize("name", sorted(CASES))
def test_halves(name, want_mass):
    c = CASES[name]
    n = len(c["pool"])
    wl = synth.make_small(71, 1, c["Hq"], c["Hkv"], c["D"], c["pool"], [list(range(len(x))) for x in c["pool"]], c["n_q"], c["n_new"], name=name)
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        _, cq, cn = wl.cu()
        for _ in range(2):                                  # the second call finds plan and pool as the first left them
            out, mass, _ = s.attend(0, q, kn, vn, want_mass=want_mass)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        p = enl.enl_plan_inspect(s.cache)
        tokens = 128 // (c["Hq"] // c["Hkv"])
        assert p["n_items"] == sum(-(-x // tokens) for x in c["n_q"]) * c["Hkv"] * p["n_splits"]
        assert p["merge_kind"] == (1 if c["splits"] else 0)
        for b in range(n):
            ro, rm, _ = s.oracle(0, b, q[cq[b]:cq[b + 1]], kn[cn[b]:cn[b + 1]], vn[cn[b]:cn[b + 1]])
            G = len(wl.sel_local[b])
            check_close(out[cq[b]:cq[b + 1]], ro, mass[cq[b]:cq[b + 1], :, :G + 1] if want_mass else None, rm if want_mass else None, what=name)


@pytest.mark.parametrize("jump", [7.0, 20.0, 65.0, 130.0])
def test_halves_of_very_different_scores(jump):
    """One half's scores lie `jump` (log2 units) above the other's, either way round: the walkers' references differ by as much."""
    for first in (True, False):
        wl = synth.make_small(72, 1, 8, 2, 128, [[256, 256]], [[0, 1] if first else [1, 0]], [40], [40], name="jump")
        with Session(wl, [0]) as s:
            q, kn, vn = wl.new_qkv(0, s.device)
            q = torch.ones_like(q) * 0.25
            step = jump / (128 * 0.25 * 1.4426950408889634 / np.sqrt(128.0))
            k, v = (x.clone() for x in wl.pool_kv(0, 0, s.device))
            k[256:] += step
            enl.enl_group_store(s.cache, 1, 0, k[256:], v[256:])
            out, mass, _ = s.attend(0, q, kn, vn)
            torch.cuda.synchronize()
            assert enl.enl_cache_status(s.cache) == enl.ENL_OK
            order = (0, 1) if first else (1, 0)
            s.host_kv[(0, 0)] = ([k[g * 256:(g + 1) * 256].cpu() for g in order], [v[g * 256:(g + 1) * 256].cpu() for g in order])
            ro, rm, _ = s.oracle(0, 0, q, kn, vn)
            check_close(out, ro, mass, rm, what=f"jump {jump}")
