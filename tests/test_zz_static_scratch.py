"""The entry point for callers that may not allocate (enl_attend_static): a robot's planner tick that
runs with memory fixed at start-up, or code hosted inside another runtime that owns the device heap,
cannot create a cache, so it hands the library one contiguous K/V buffer and the library keeps its
split-KV partials in a device array that is part of the library image.  Its result must equal what the
allocating path (enl_attend with one query token over the same groups) returns, call after call: the
built-in array is shared by all calls and still holds the previous call's partials."""
import numpy as np
import pytest
import torch

from oracle import enl_oracle as orc
from paper_2510_18546_b200 import enl, synth
from tests.helpers import MASS_MAX_ABS, OUT_MAX_ABS, OUT_MEAN_ABS, Session, check_close

pytestmark = pytest.mark.gpu


def both_paths(s, wl, sel, t, want_mass=True):
    """(out, mass) of enl_attend (n_q = 1, n_new = t + 1) and of enl_attend_static on the same keys."""
    q, kn, vn = wl.new_qkv(0, s.device)
    out_a, mass_a, _ = s.attend(0, q[t:t + 1], kn[:t + 1], vn[:t + 1], n_q=[1], n_new=[t + 1], sel_override=sel)
    k, v = wl.pool_kv(0, 0, s.device)
    offs = wl.pool_offsets(0)
    ks = [k[offs[g]:offs[g + 1]] for g in sel] + [kn[:t + 1]]
    vs = [v[offs[g]:offs[g + 1]] for g in sel] + [vn[:t + 1]]
    kc, vc = torch.cat(ks).contiguous(), torch.cat(vs).contiguous()
    out_s = torch.full((wl.n_q_heads, wl.head_dim), float("nan"), dtype=torch.bfloat16, device=s.device)
    mass_s = torch.full((wl.n_q_heads, len(sel) + 1), float("nan"), dtype=torch.float32, device=s.device) if want_mass else None
    enl.enl_attend_static([int(wl.pool_lens[0][g]) for g in sel], t + 1, q[t], kc, vc, out_s, mass_s,
                          stream=torch.cuda.current_stream(s.device).cuda_stream)
    torch.cuda.synchronize()
    # the float64 oracle on the same contiguous keys, the segments as its slots: a mistake shared by the two
    # one-token CUDA paths would pass a comparison of one with the other
    ro, rm = orc.attend_slots(wl.n_q_heads, wl.n_kv_heads, wl.head_dim, [x.cpu() for x in ks[:-1]],
                              [x.cpu() for x in vs[:-1]], q[t:t + 1].cpu(), kn[:t + 1].cpu(), vn[:t + 1].cpu())
    check_close(out_s[None], ro, mass_s[None] if want_mass else None, rm if want_mass else None, "static vs oracle")
    return out_a[0], (mass_a[0, :, :len(sel) + 1] if want_mass else None), out_s, mass_s


def assert_same(out_a, mass_a, out_s, mass_s):
    err = (out_a.float() - out_s.float()).abs()
    assert torch.isfinite(out_s.float()).all()
    assert err.max().item() <= OUT_MAX_ABS and err.mean().item() <= OUT_MEAN_ABS
    if mass_a is not None:
        assert torch.isfinite(mass_s).all()
        assert (mass_a - mass_s).abs().max().item() <= MASS_MAX_ABS
        assert (mass_s.sum(-1) - 1).abs().max().item() <= MASS_MAX_ABS


def test_two_calls_in_a_row_match_the_allocating_path():
    wl = synth.make_small(31, 1, 32, 8, 128, [[300, 17, 256, 90, 0, 1200]], [[0, 1, 2, 3, 4, 5]], [40], [40],
                          sigma=0.5, name="static")
    with Session(wl, [0]) as s:
        # first call: many keys, many splits; second call: fewer segments and keys, so stale partials of the
        # first call sit right behind what the second one writes
        assert_same(*both_paths(s, wl, [5, 0, 4, 2, 1, 3], 39))
        assert_same(*both_paths(s, wl, [1, 3], 0))
        assert_same(*both_paths(s, wl, [], 7))
        assert_same(*both_paths(s, wl, [5, 2], 20, want_mass=False))


def test_head_dim_64_and_other_head_ratios():
    wl = synth.make_small(32, 1, 8, 2, 64, [[33, 70, 18, 5]], [[0, 1, 2, 3]], [12], [12], name="static64")
    with Session(wl, [0]) as s:
        assert_same(*both_paths(s, wl, [2, 0, 3, 1], 11))
        assert_same(*both_paths(s, wl, [3], 0))


def test_limits_are_reported_not_enqueued():
    dev = torch.device("cuda:0")
    q = torch.zeros(32, 128, dtype=torch.bfloat16, device=dev)
    kv = torch.zeros(64, 8, 128, dtype=torch.bfloat16, device=dev)
    out = torch.zeros_like(q)
    with pytest.raises(enl.EnlError) as e:       # more keys than ENL_STATIC_MAX_KEYS (sizes only; nothing is read)
        enl.enl_attend_static([enl.ENL_STATIC_MAX_KEYS], 1, q, kv, kv, out)
    assert e.value.code == enl.ENL_E_LIMIT
    with pytest.raises(enl.EnlError) as e:       # more segments than ENL_STATIC_MAX_SEGMENTS
        enl.enl_attend_static([0] * (enl.ENL_STATIC_MAX_SEGMENTS + 1), 1, q, kv, kv, out)
    assert e.value.code == enl.ENL_E_LIMIT
    q16 = torch.zeros(32, 128, dtype=torch.bfloat16, device=dev)
    kv1 = torch.zeros(64, 2, 128, dtype=torch.bfloat16, device=dev)
    with pytest.raises(enl.EnlError) as e:       # 16 q heads per kv head
        enl.enl_attend_static([10], 1, q16, kv1, kv1, out)
    assert e.value.code == enl.ENL_E_LIMIT
    with pytest.raises(enl.EnlError) as e:
        enl.enl_attend_static([10], 0, q, kv, kv, out)
    assert e.value.code == enl.ENL_E_INVAL


def rounded(p, terms):
    """p as the sum of its first `terms` bf16 terms."""
    got = np.zeros_like(p)
    for _ in range(terms):
        got += torch.tensor(p - got).to(torch.bfloat16).double().numpy()
    return got


@pytest.mark.parametrize("path", ["cluster", "general"])
@pytest.mark.parametrize("D", [64, 128])
def test_probabilities_are_fp32(D, path):
    """Three neighbouring keys whose values all but cancel: v_b = -bf16(v_a p_a / p_b), v_c = -bf16 of what that leaves.  The rest
    is some 2^-18 of v_a, so an output shows how exactly the probabilities went into the product: with two bf16 terms of them (17
    bits) it is wrong altogether, while fp32 arithmetic keeps it within a few per cent."""
    Hq, Hkv, seg, n_new, dev = 8, 2, [16, 5, 33], 10, torch.device("cuda:0")
    n = sum(seg) + n_new
    gen = torch.Generator().manual_seed(D)
    q = torch.randn(Hkv, 1, D, generator=gen).repeat(1, Hq // Hkv, 1).reshape(Hq, D).to(torch.bfloat16)      # all heads of a kv head agree
    k = (0.7 * torch.randn(n, Hkv, D, generator=gen)).to(torch.bfloat16)
    v = (1.0 + torch.rand(n, Hkv, D, generator=gen)).to(torch.bfloat16)
    s = np.einsum("hd,nhd->hn", q.reshape(Hkv, -1, D)[:, 0].double().numpy(), k.double().numpy()) / np.sqrt(D)
    p = np.exp(s - s.max(axis=1, keepdims=True))
    p /= p.sum(axis=1, keepdims=True)
    ends = np.cumsum([0] + seg + [n_new])
    pages = [(i, min(i + 16, e)) for a, e in zip(ends, ends[1:]) for i in range(a, e, 16)]
    for a, e in pages:                                           # the three are of one page, so that one warp adds them up
        v[a + (e - a) // 3 * 3:e] = 0                            # keys without partners
        for i in range(a, e - 2, 3):
            rest = v[i].double()                                 # what key i (then i + 1) leaves, in units of the next key's probability
            for j in (i + 1, i + 2):
                rest = rest * torch.tensor(p[:, j - 1] / p[:, j])[:, None]
                v[j] = (-rest).to(torch.bfloat16)
                rest = rest + v[j].double()
    vd = v.double().numpy()
    ks, vs = ([x[a:e] for a, e in zip(ends[:-2], ends[1:-1])] for x in (k, v))
    want, _ = orc.attend_slots(Hq, Hkv, D, ks, vs, q[None], k[ends[-2]:], v[ends[-2]:])
    want = want.reshape(Hkv, -1, D)[:, 0]
    size = np.linalg.norm(want)
    # one bf16 rounding of the output; scores (products and sums in fp32), ex2 and the sums of the second product each err by
    # about 2^-23 of a probability, independently from key to key
    bound = 2.0 ** -9 + 2.0 ** -21 * np.linalg.norm(np.sqrt(np.einsum("hn,nhd->hd", p ** 2, vd ** 2))) / size
    for terms, enough in ((1, False), (2, False), (3, True)):
        err = np.linalg.norm(np.einsum("hn,nhd->hd", rounded(p, terms), vd) - want) / size
        assert (err < bound / 8) if enough else (err > 1.5 * bound), (terms, err, bound)
    out = torch.empty(Hq, D, dtype=torch.bfloat16, device=dev)
    flat = torch.empty(2, n * Hkv * D + 8, dtype=torch.bfloat16, device=dev)
    at = 0 if path == "cluster" else 1                           # tensors off the 16-byte boundary take the general kernels
    kd, vv = (x[at:at + n * Hkv * D].view(n, Hkv, D) for x in flat)
    kd.copy_(k), vv.copy_(v)
    enl.enl_attend_static(seg, n_new, q.to(dev), kd, vv, out, None)
    torch.cuda.synchronize()
    assert enl.enl_static_status() == enl.ENL_OK
    got = out.double().cpu().numpy().reshape(Hkv, -1, D)
    for h in range(Hq // Hkv):
        err = np.linalg.norm(got[:, h] - want) / size
        assert err <= bound, (h, err, bound)
