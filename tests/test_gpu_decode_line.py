"""One-token steps on both sides of the lines from which on a stream is long enough for the streaming kernel."""
import pytest
import torch

from paper_2510_18546_b200 import enl, synth
from tests.helpers import Session, check_close

pytestmark = pytest.mark.gpu

# (q heads, kv heads, head_dim, pages per CTA at the line, CTAs per cluster, episodes)
LINES = [(32, 8, 128, 64, 16, 1), (8, 2, 128, 88, 16, 1), (32, 8, 64, 112, 16, 1), (16, 8, 128, 88, 8, 2)]


@pytest.mark.parametrize("want_mass", [True, False])
@pytest.mark.parametrize("above", [False, True])
@pytest.mark.parametrize("line", LINES)
def test_step_at_the_line(line, above, want_mass):
    hq, hkv, d, pages, ctas, n = line
    keys = 16 * (pages * ctas + (8 if above else -8))       # pages of the stream are counted in eights; the new token has one of its own
    wl = synth.make_small(81, 1, hq, hkv, d, [[keys // 3, keys - keys // 3 - 100, 100]] * n, [[0, 1, 2]] * n, [1] * n, [1] * n, name="line")
    with Session(wl, [0]) as s:
        q, kn, vn = wl.new_qkv(0, s.device)
        out, mass, _ = s.attend(0, q, kn, vn, want_mass=want_mass)
        torch.cuda.synchronize()
        assert enl.enl_cache_status(s.cache) == enl.ENL_OK and enl.enl_plan_inspect(s.cache)["merge_kind"] == 3
        for b in range(n):
            ro, rm, _ = s.oracle(0, b, q[b:b + 1], kn[b:b + 1], vn[b:b + 1])
            check_close(out[b:b + 1], ro, mass[b:b + 1] if want_mass else None, rm if want_mass else None, what=f"line {line}")
