"""Masses finished by a launch of their own, just below and above the grid size (four CTAs per multiprocessor) where it keeps sixteen or eight loads in flight:
with outputs (no splits), without (key ranges split), with the objects' sums."""
import pytest
import torch

from paper_2510_18546_b200 import enl, synth
from tests.helpers import MASS_MAX_ABS, Session

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mass_only", [False, True])
@pytest.mark.parametrize("over", [-3, 0, 1])                # the last row block below the line ragged or full; a row beyond it
def test_masses_around_the_line(over, mass_only):
    # a CTA finishes 8 rows x 32 heads and 32 slots, so five CTAs are one row block over the 131 slots
    n_q = 4 * torch.cuda.get_device_properties(0).multi_processor_count // 5 * 8 + over
    sizes = [1 + (i * 5) % 3 for i in range(130)]           # five slot blocks
    wl = synth.make_small(73, 1, 32, 8, 64, [sizes], [list(range(130))], [n_q], [n_q], name="finish")
    cuts = [0, 1, n_q // 3, n_q - 40]                       # the last rows belong to no object
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        out = None if mass_only else torch.empty(n_q, 32, 64, dtype=torch.bfloat16, device=s.device)
        mass = torch.full((n_q, 32, 131), float("nan"), device=s.device)
        sums = torch.zeros(len(cuts) - 1, 131, device=s.device)
        enl.enl_attend(s.cache, 0, wl.sel_ids(), q, kn, vn, out, mass, flags=enl.ENL_MASS_ONLY if mass_only else 0, group_mass_sum=sums, obj_off=cuts)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK
        rows = [0, 1, n_q // 3, n_q - 41, n_q - 2, n_q - 1]
        _, ref, _ = s.oracle(0, 0, q, kn, vn, rows=rows)
        m = mass.double().cpu()
        assert torch.isfinite(m).all()
        assert (m.sum(-1) - 1).abs().max() <= 131 * MASS_MAX_ABS
        assert (m[rows] - torch.as_tensor(ref)).abs().max() <= MASS_MAX_ABS
        for o in range(len(cuts) - 1):
            want = m[cuts[o]:cuts[o + 1]].sum((0, 1))
            # fp32 sums of n addends that are not negative: relative error below n * 2^-24
            n = (cuts[o + 1] - cuts[o]) * 32
            assert ((sums[o].double().cpu() - want).abs() <= want * n * 2.0 ** -24 + 1e-30).all()
