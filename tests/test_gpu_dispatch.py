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
